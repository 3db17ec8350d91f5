// Monitoring kernel: per-token Kullback-Leibler divergences between the
// full-vocabulary inference and training policies and their entropies (the
// stability metric of Sec. 6; the entropy Sec. 7 proposes to adapt rho to).
//
// Both rows are streamed together, once, in 32-byte granules, two of each in flight per thread.  Each thread
// keeps, for each policy, an online log-sum-exp state in the base-2 domain extended by two weighted sums:
// with w_k = 2^{z_k l - c},
//   s = sum w_k,  a = sum w_k z_k,  b = sum w_k (z'_k - z_k),
// from which  H = lse - a / s,  KL(train || infer) = -b/s - lse + lse',
// KL(infer || train) = b'/s' - lse' + lse.
//
// Two logits go through one instruction (f32x2) and two granules through one check of the running maximum: with a
// dozen instructions for every pair of logits the kernel is bound by issue and by its exponentials (0.7 of the
// time that the bytes take), not by HBM.  T = 4096 x V = 151,936 bfloat16, 2.49 GB, in bursts in turn with the form
// that takes one logit an instruction: 483 -> 450 us (386 at the copy bandwidth); 1,000 x 50,021 with rows back to
// back, element by element there: 129 -> 46.  Blocks per SM: bfloat16 446 / 459 at 4 / 3, float32 (2,000 x 262,144)
// 661 / 606.  Loads of the next granules before the last ones are worked on are slower (few rows 31 against 23 us,
// 4,096 rows 487 against 450): the code spills or runs with fewer warps.  One reference for the whole block, below
// the maximum, loses the divergence of rows with one dominant token (float32, V = 5,000, heavy-tailed: relative error
// 3.6e-3 against 3.7e-4).
//
// Accuracy against float64, relative 2-norm over a batch: entropies 1e-6 to 2e-6 (one dominant token and heavy tails,
// where the entropy itself is small: 2e-5 to 1e-4); divergences are differences of sums of order one, good to some
// 2e-7 absolute, 1e-3 relative where they are 2e-4.
#include "dvp_rows_impl.cuh"

namespace dvp {

struct Moments {
  float m, c, s, a, b;
};

__device__ __forceinline__ Moments combine(const Moments &x, const Moments &y) {
  Moments r;
  r.m = fmaxf(x.m, y.m);
  r.c = fmaxf(x.c, y.c);
  const float fx = x.c > kNegInf ? ex2(x.c - r.c) : 0.f;
  const float fy = y.c > kNegInf ? ex2(y.c - r.c) : 0.f;
  r.s = x.s * fx + y.s * fy;
  r.a = x.a * fx + y.a * fy;
  r.b = x.b * fx + y.b * fy;
  return r;
}

__device__ __forceinline__ Moments shfl_xor(const Moments &v, int o) {
  Moments r;
  r.m = __shfl_xor_sync(0xffffffffu, v.m, o);
  r.c = __shfl_xor_sync(0xffffffffu, v.c, o);
  r.s = __shfl_xor_sync(0xffffffffu, v.s, o);
  r.a = __shfl_xor_sync(0xffffffffu, v.a, o);
  r.b = __shfl_xor_sync(0xffffffffu, v.b, o);
  return r;
}

// scratch: 5 x 32 floats.  Fixed order; the result is valid in every thread.
__device__ __forceinline__ Moments block_reduce(Moments v, float *scratch) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = (blockDim.x + 31) >> 5;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const Moments other = shfl_xor(v, o);
    v = (lane & o) ? combine(other, v) : combine(v, other);
  }
  __syncthreads();
  if (lane == 0) {
    scratch[warp] = v.m;
    scratch[32 + warp] = v.c;
    scratch[64 + warp] = v.s;
    scratch[96 + warp] = v.a;
    scratch[128 + warp] = v.b;
  }
  __syncthreads();
  Moments r = {kNegInf, kNegInf, 0.f, 0.f, 0.f};
  if (lane < nwarp) {
    r.m = scratch[lane];
    r.c = scratch[32 + lane];
    r.s = scratch[64 + lane];
    r.a = scratch[96 + lane];
    r.b = scratch[128 + lane];
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const Moments other = shfl_xor(r, o);
    r = (lane & o) ? combine(other, r) : combine(r, other);
  }
  return r;
}

// The sums of one policy, as pairs: of the even and of the odd elements.
struct PairSums {
  uint64_t s, a, b;

  // two logits x, d = z' - z of both, reference c
  __device__ __forceinline__ void absorb(uint64_t x, uint64_t d, float c) {
    float w0, w1;
    unpack2(fma2(x, pack2(kLog2e, kLog2e), pack2(-c, -c)), w0, w1);
    const uint64_t w = pack2(ex2(w0), ex2(w1));
    s = add2(s, w);
    a = fma2(w, x, a);
    b = fma2(w, d, b);
  }
  __device__ __forceinline__ void add(const PairSums &q) {
    s = add2(s, q.s);
    a = add2(a, q.a);
    b = add2(b, q.b);
  }
};

// The state of one policy over a thread's elements.  The maximum itself is kept for float32 logits only: with 2-byte
// logits the register is worth more (64 x 151,936: 24.6 -> 22.6 us; T = 4096: 471 -> 453), with float32 ones the code
// without it spills (2,500 x 100,000: 310 against 314 us).
template <typename TIn>
struct PairMoments {
  static constexpr bool kKeepMax = sizeof(TIn) == 4;
  float m, c;
  PairSums q;

  // Move the reference to a larger maximum.
  __device__ __forceinline__ void raise(float new_max) {
    if constexpr (kKeepMax) {
      if (new_max > m) {
        rescale(log2_reference(new_max));
        m = new_max;
      }
    } else {
      const float cn = log2_reference(new_max);
      if (cn > c) rescale(cn);
    }
  }
  __device__ __forceinline__ void rescale(float cn) {
    const float f = ex2(c - cn);  // c = -inf at the start: factor 0
    const uint64_t f2 = pack2(f, f);
    q.s = mul2(q.s, f2);
    q.a = mul2(q.a, f2);
    q.b = mul2(q.b, f2);
    c = cn;
  }
  __device__ __forceinline__ Moments sum() const {
    Moments r = {kKeepMax ? m : c / kLog2e, c, 0.f, 0.f, 0.f};  // m: to float32 rounding, for a correction of 1e-8 of it
    float lo, hi;
    unpack2(q.s, lo, hi);
    r.s = lo + hi;
    unpack2(q.a, lo, hi);
    r.a = lo + hi;
    unpack2(q.b, lo, hi);
    r.b = lo + hi;
    return r;
  }
};

__device__ __forceinline__ uint64_t difference(uint64_t x, uint64_t y) { return fma2(x, pack2(-1.f, -1.f), y); }

template <typename TIn>
__device__ __forceinline__ void absorb_granules(const Granule<TIn> &gt, const Granule<TIn> &gi, float ca, float cb,
                                                PairSums &a, PairSums &b) {
  constexpr int kElems = Granule<TIn>::kElems;
  float x[kElems], y[kElems];
  gt.get(x);
  gi.get(y);
#pragma unroll
  for (int j = 0; j < kElems; j += 2) {
    const uint64_t xx = pack2(x[j], x[j + 1]), yy = pack2(y[j], y[j + 1]), d = difference(xx, yy);
    a.absorb(xx, d, ca);
    b.absorb(yy, d, cb);
  }
}

// The largest element of two granules.
template <typename TIn>
__device__ __forceinline__ float max_of(const Granule<TIn> &g, const Granule<TIn> &h) {
  if constexpr (sizeof(TIn) == 4) {
    return fmaxf(g.max(), h.max());
  } else {
    return SweepOps<TIn>::value(__hmax2(SweepOps<TIn>::tree(g), SweepOps<TIn>::tree(h)));
  }
}

// One element of each row, under references that are at least as large.
template <typename TIn>
__device__ __forceinline__ void absorb_one(float x, float y, PairMoments<TIn> &a, PairMoments<TIn> &b) {
  // the pair's other element: -inf has no weight, but it may not be multiplied
  const float wa = ex2(fmaf(x, kLog2e, -a.c)), wb = ex2(fmaf(y, kLog2e, -b.c)), d = y - x;
  const uint64_t wa2 = pack2(wa, 0.f), wb2 = pack2(wb, 0.f), d2 = pack2(d, 0.f);
  a.q.s = add2(a.q.s, wa2);
  a.q.a = fma2(wa2, pack2(x, 0.f), a.q.a);
  a.q.b = fma2(wa2, d2, a.q.b);
  b.q.s = add2(b.q.s, wb2);
  b.q.a = fma2(wb2, pack2(y, 0.f), b.q.a);
  b.q.b = fma2(wb2, d2, b.q.b);
}

struct MonitorParams {
  const void *train, *infer;
  long long T, V, ld_train, ld_infer;
  float *kl_it, *kl_ti, *h_t, *h_i;
  unsigned int *bounds_status;  // the bounds-checking build's status word; unused otherwise
};

__device__ __forceinline__ void monitor_finish(const MonitorParams &p, long long t, const Moments &a,
                                               const Moments &b) {
  const double ln2 = 0.6931471805599453094;
  const double corr = 1.0 - (double)kLog2e * ln2;
  const double lse_t = ln2 * ((double)a.c + (double)log2f(a.s)) + corr * (double)a.m;
  const double lse_i = ln2 * ((double)b.c + (double)log2f(b.s)) + corr * (double)b.m;
  const double ez_t = (double)a.a / (double)a.s, ed_t = (double)a.b / (double)a.s;
  const double ez_i = (double)b.a / (double)b.s, ed_i = (double)b.b / (double)b.s;
  if (p.kl_ti) p.kl_ti[t] = (float)(-ed_t - lse_t + lse_i);
  if (p.kl_it) p.kl_it[t] = (float)(ed_i - lse_i + lse_t);
  if (p.h_t) p.h_t[t] = (float)(lse_t - ez_t);
  if (p.h_i) p.h_i[t] = (float)(lse_i - ez_i);
}

// How a block reads its two rows.  kLong, kShort: the rows of a token start alike against the 32-byte grid; granules are
// cut at the rows' own boundaries, the elements in front of the first and behind the last whole granule are taken one
// per thread.  kShort (several steps of 64 threads, up to 16 granules of each row a thread): every step's terms are
// added up by themselves first, because 64 threads add four times as many terms one after the other as the 256 that
// such a row had once (V = 15,000 float16: relative error of KL 1.30e-3 -> 1.12e-3, of the entropy 2.8e-6 -> 1.5e-6;
// 5,000 x 16,000 bfloat16 70 / 68 us, 20,000 x 4,000 94 / 97).  kElementwise: any rows, in two passes.
enum class Rows { kElementwise, kShort, kLong, kShared };
//
// kShared: kLong with the rows of a token shared by the 2^log_parts blocks of a cluster, for few rows: each takes its part
// of the granules, and the first adds up what the others leave in their shared memory.  (4 x 151,936 bfloat16 22.5 -> 10.2
// us, 45 x 225,920 30.7 -> 18.4, 64 x 151,936 22.5 -> 18.4; float32 26.3 / 34.9 / 26.6 -> 10.3 / 18.4 / 22.9.)
template <typename TIn, Rows kRows>
__global__ void __launch_bounds__(256, sizeof(TIn) == 2 && kRows != Rows::kShort ? 4 : 3)
dvp_monitor_kernel(const MonitorParams p, const int log_parts) {
  __shared__ float scratch[160];
  constexpr int kElems = Granule<TIn>::kElems;
  const long long t = kRows == Rows::kShared ? blockIdx.x >> log_parts : blockIdx.x;
  const int part = kRows == Rows::kShared ? (int)blockIdx.x & ((1 << log_parts) - 1) : 0;
  const TIn *zt = reinterpret_cast<const TIn *>(p.train) + t * p.ld_train;
  const TIn *zi = reinterpret_cast<const TIn *>(p.infer) + t * p.ld_infer;
  const int V = (int)p.V, tid = (int)threadIdx.x, n_thr = (int)blockDim.x;
  PairMoments<TIn> a = {kNegInf, kNegInf, {0, 0, 0}}, b = a;
  if constexpr (kRows != Rows::kElementwise) {
    const int mis = (int)(((uintptr_t)zt & 31u) / sizeof(TIn));
    const int head = min(V, mis ? kElems - mis : 0), n_full = (V - head) / kElems;
    DVP_BOUNDS_BEGIN(p.bounds_status);
    DVP_BOUNDS_SET(n_gran, n_full);
    DVP_BOUNDS_SET(V, (long long)n_full * kElems);
    DVP_BOUNDS_SYNC();
    const TIn *bt = zt + head, *bi = zi + head;
    const int per = kRows == Rows::kShared ? (n_full + (1 << log_parts) - 1) >> log_parts : n_full;
    const int g_end = kRows == Rows::kShared ? min(n_full, (part + 1) * per) : n_full;
    for (int g = part * per + tid; g < g_end; g += 2 * n_thr) {
      Granule<TIn> t0, i0, t1, i1;
      const int g1 = g + n_thr;
      if (!DVP_IN((long long)g * kElems + kElems - 1, V, DVP_OOB_GLOBAL)) break;
      const bool second = g1 < g_end && DVP_IN((long long)g1 * kElems + kElems - 1, V, DVP_OOB_GLOBAL);
      t0.load(bt + (size_t)g * kElems);
      i0.load(bi + (size_t)g * kElems);
      t1.load(bt + (size_t)(second ? g1 : g) * kElems);
      i1.load(bi + (size_t)(second ? g1 : g) * kElems);
      a.raise(max_of<TIn>(t0, t1));
      b.raise(max_of<TIn>(i0, i1));
      if constexpr (kRows == Rows::kShort) {
        PairSums pa = {0, 0, 0}, pb = pa;
        absorb_granules<TIn>(t0, i0, a.c, b.c, pa, pb);
        if (second) absorb_granules<TIn>(t1, i1, a.c, b.c, pa, pb);
        a.q.add(pa);
        b.q.add(pb);
      } else {
        absorb_granules<TIn>(t0, i0, a.c, b.c, a.q, b.q);
        if (second) absorb_granules<TIn>(t1, i1, a.c, b.c, a.q, b.q);
      }
    }
    const int k = tid < head ? tid : tid + n_full * kElems;  // fewer than 64 of them
    if (k < V && part == 0) {
      const float x = Storage<TIn>::widen(zt[k]), y = Storage<TIn>::widen(zi[k]);
      a.raise(x);
      b.raise(y);
      absorb_one(x, y, a, b);
    }
  } else {
    float mt = kNegInf, mi = kNegInf;
    for (long long k = tid; k < p.V; k += n_thr) {
      mt = fmaxf(mt, Storage<TIn>::widen(zt[k]));
      mi = fmaxf(mi, Storage<TIn>::widen(zi[k]));
    }
    a.raise(mt);
    b.raise(mi);
    // the maximum is known: no reference moves in this pass, and two elements go through one instruction (bfloat16
    // 700 x 20,000: 46 -> 33 us, 1,000 x 50,021: 167 -> 124; float32 700 x 20,000: 58 -> 43)
    long long k = tid;
    for (; k + n_thr < p.V; k += 2 * n_thr) {
      const uint64_t xx = pack2(Storage<TIn>::widen(zt[k]), Storage<TIn>::widen(zt[k + n_thr]));
      const uint64_t yy = pack2(Storage<TIn>::widen(zi[k]), Storage<TIn>::widen(zi[k + n_thr]));
      const uint64_t d = difference(xx, yy);
      a.q.absorb(xx, d, a.c);
      b.q.absorb(yy, d, b.c);
    }
    if (k < p.V) absorb_one(Storage<TIn>::widen(zt[k]), Storage<TIn>::widen(zi[k]), a, b);
  }
  Moments ra = block_reduce(a.sum(), scratch);
  Moments rb = block_reduce(b.sum(), scratch);
  if constexpr (kRows == Rows::kShared) {
    __shared__ float left[10];
    if (tid == 0) {
      const float v[10] = {ra.m, ra.c, ra.s, ra.a, ra.b, rb.m, rb.c, rb.s, rb.a, rb.b};
#pragma unroll
      for (int i = 0; i < 10; ++i) left[i] = v[i];
    }
    cluster_arrive();
    cluster_wait();
    if (part == 0 && tid == 0) {
      for (uint32_t k = 1; k < 1u << log_parts; ++k) {  // in order
        float v[10];
#pragma unroll
        for (int i = 0; i < 10; ++i) v[i] = ld_cluster_f32(left + i, k);
        ra = combine(ra, {v[0], v[1], v[2], v[3], v[4]});
        rb = combine(rb, {v[5], v[6], v[7], v[8], v[9]});
      }
    }
    cluster_arrive();  // no block leaves before its sums are read
    cluster_wait();
  }
  if (part == 0 && tid == 0) monitor_finish(p, t, ra, rb);
}

template <typename TIn>
static cudaError_t launch_monitor(const MonitorParams &p, cudaStream_t s) {
  const long long elem = sizeof(TIn);
  const bool alike = ((long long)((uintptr_t)p.train % 32) - (long long)((uintptr_t)p.infer % 32)) % 32 == 0 &&
                     (p.T == 1 || (p.ld_train - p.ld_infer) * elem % 32 == 0);
  if (!alike) {
    dvp_monitor_kernel<TIn, Rows::kElementwise><<<(unsigned)p.T, 256, 0, s>>>(p, 0);
    return cudaGetLastError();
  }
  // some 16 granules of each row a thread, as in the row kernels
  const long long n_gran = p.V * elem / 32;
  int threads = 64, log_parts = 0;
  while (threads < 256 && 16LL * threads < n_gran) threads *= 2;
  while (threads < 256 && 2 * p.T * threads <= 148 * 1024) threads *= 2;
  // several blocks a token while all of them fit the chip at once, with a step and a half or more each
  while (log_parts < 3 && (p.T << (log_parts + 1)) * threads <= 148 * 1024 && n_gran >> (log_parts + 1) >= 3 * threads)
    ++log_parts;
  if (log_parts == 0) {
    if (threads == 64 && n_gran > 2 * threads)
      dvp_monitor_kernel<TIn, Rows::kShort><<<(unsigned)p.T, threads, 0, s>>>(p, 0);
    else
      dvp_monitor_kernel<TIn, Rows::kLong><<<(unsigned)p.T, threads, 0, s>>>(p, 0);
    return cudaGetLastError();
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(p.T << log_parts), 1, 1);
  cfg.blockDim = dim3((unsigned)threads, 1, 1);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 1u << log_parts;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, dvp_monitor_kernel<TIn, Rows::kShared>, p, log_parts);
}

}  // namespace dvp

extern "C" int dvp_monitor(const dvp_monitor_args *a) {
  if (!a || a->struct_size != sizeof(dvp_monitor_args)) return DVP_ERR_INVALID_ARG;
  if (a->logits_dtype != DVP_F32 && a->logits_dtype != DVP_BF16 && a->logits_dtype != DVP_F16)
    return DVP_ERR_UNSUPPORTED;
  if (a->T < 0 || a->T > 0x7fffffffLL || a->V < 1) return DVP_ERR_INVALID_ARG;
  if (a->V > 0x7fffff00LL) return DVP_ERR_UNSUPPORTED;
  if (a->T == 0) return DVP_OK;
  if (!a->train_logits || !a->infer_logits || a->ld_train < a->V || a->ld_infer < a->V)
    return DVP_ERR_INVALID_ARG;
  dvp::MonitorParams p{a->train_logits, a->infer_logits, a->T, a->V, a->ld_train, a->ld_infer,
                       a->kl_infer_train, a->kl_train_infer, a->entropy_train, a->entropy_infer,
                       dvp::bounds_status_word()};
  cudaStream_t s = static_cast<cudaStream_t>(a->stream);
  cudaError_t e;
  switch (a->logits_dtype) {
    case DVP_F32: e = dvp::launch_monitor<float>(p, s); break;
    case DVP_BF16: e = dvp::launch_monitor<__nv_bfloat16>(p, s); break;
    default: e = dvp::launch_monitor<__half>(p, s); break;
  }
  return e == cudaSuccess ? DVP_OK : DVP_ERR_CUDA;
}
