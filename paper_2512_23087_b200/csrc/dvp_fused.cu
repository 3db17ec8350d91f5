// Fused LM-head entry point: z = hidden x W_vocab^T on the tensor cores, the
// row computation of dvp_forward on panels of those logits, and the chain rule
// through the head (d_hidden = G W, d_w = G^T hidden) as two more contractions.
//
// The [T, V] training logits are never stored: a panel of `panel_rows` tokens
// lives in the workspace as fp32 logits, is read once by the panel's row pass
// (dvp_panel.cuh), which leaves the per-token results and the gradient panel up to
// one factor per row, and that panel is consumed by the two gradient contractions
// before the next panel overwrites it.
//
// The panel is held in float16 (11-bit significand; bfloat16's 8 bits would miss
// the 1e-3 gradient tolerance by themselves): P = 2^14 e^{z - m} on the safe set.
// The factor per row, -g / (2^14 s_S), multiplies the rows of d_hidden in the
// contraction's epilogue and, times a power of two chosen from max |upstream|, the
// hidden rows as they are converted to float16 for the d_w contraction; the inverse
// power of two is applied in that contraction's epilogue.  tcgen05 kind::f16 needs
// both operands of one type, so W is converted to a float16 copy once per call
// (exact for bfloat16 values in float16's normal range).
#include <cmath>
#include <mutex>

#include "dvp_common.cuh"
#include "dvp_gemm.cuh"
#include "dvp_panel.cuh"

namespace dvp {

// out[c, r] = convert(in[r, c]) for a row-major [R, C] input of a 16-bit type.
// 64 x 64 tiles through shared memory; 16-byte accesses on both sides when the
// strides and bases allow it (ld_in, ld_out multiples of 8, 16-byte aligned bases).
template <typename TIn, typename TOut>
__global__ void __launch_bounds__(256)
transpose_convert_kernel(const TIn *in, long long ld_in, TOut *out, long long ld_out, int R, int C,
                         int vec_ok, const float *row_scale) {
  __shared__ TOut tile[64][66];
  begin_after(true);
  const int per_row = (C + 63) / 64, c0 = (int)(blockIdx.x % per_row) * 64, r0 = (int)(blockIdx.x / per_row) * 64;
  const int tid = threadIdx.x;
  // load: 64 rows x 8 vectors of 8 elements, two vectors per thread
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const int v = tid + i * 256, r = r0 + (v >> 3), c = c0 + (v & 7) * 8;
    TOut e[8];
    const float rs = (row_scale && r < R) ? row_scale[r] : 1.f;  // input row r times rs
    if (vec_ok && r < R && c + 8 <= C) {
      const uint4 raw = *reinterpret_cast<const uint4 *>(in + (long long)r * ld_in + c);
      const TIn *x = reinterpret_cast<const TIn *>(&raw);
#pragma unroll
      for (int j = 0; j < 8; ++j) e[j] = Storage<TOut>::narrow(Storage<TIn>::widen(x[j]) * rs);
    } else {
#pragma unroll
      for (int j = 0; j < 8; ++j)
        e[j] = (r < R && c + j < C)
                   ? Storage<TOut>::narrow(Storage<TIn>::widen(in[(long long)r * ld_in + c + j]) * rs)
                   : Storage<TOut>::narrow(0.f);
    }
#pragma unroll
    for (int j = 0; j < 8; ++j) tile[v >> 3][(v & 7) * 8 + j] = e[j];
  }
  __syncthreads();
  // store: 64 output rows (input columns) x 8 vectors of 8 input rows
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const int v = tid + i * 256, c = c0 + (v >> 3), r = r0 + (v & 7) * 8;
    if (c >= C) continue;
    __align__(16) TOut e[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) e[j] = tile[(v & 7) * 8 + j][v >> 3];
    TOut *dst = out + (long long)c * ld_out + r;
    if (vec_ok && r + 8 <= R) {
      *reinterpret_cast<uint4 *>(dst) = *reinterpret_cast<const uint4 *>(e);
    } else {
      for (int j = 0; j < 8 && r + j < R; ++j) dst[j] = e[j];
    }
  }
  if (blockIdx.x == gridDim.x - 1 && tid == 0) end_after(true);  // the others leave their place to the next blocks
}

template <typename TIn, typename TOut>
static void launch_transpose(const TIn *in, long long ld_in, TOut *out, long long ld_out, int R, int C,
                             cudaStream_t s, const float *row_scale = nullptr) {
  const int vec_ok = ld_in % 8 == 0 && ld_out % 8 == 0 && (uintptr_t)in % 16 == 0 && (uintptr_t)out % 16 == 0;
  (void)launch_after(transpose_convert_kernel<TIn, TOut>, (unsigned)(((C + 63) / 64) * (long long)((R + 63) / 64)), 256, 0,
                     s, in, ld_in, out, ld_out, R, C, vec_ok, row_scale);
}

struct FusedScalars {
  int status;       // non-zero when a tensor-core kernel gave up waiting
  float scale;      // power of two applied to the gradient panel
  float inv_scale;  // its inverse
};

// What a block beside a pair contraction's may take of shared memory: an SM that holds the latter alone is set to 196 KB, of which
// every block takes 1 KB more than it asks for.  grad_scale's scratch is all that to_half_kernel has.
constexpr size_t kBesidePair = 196 * 1024 - (gemm::kSmemBytes2 + 1024) - 1024;
constexpr int kScaleFloats = 32;
static_assert(kScaleFloats * sizeof(float) <= kBesidePair, "to_half_kernel's blocks fit beside the first contraction's");

// scale = 2^(14 - x) with max|g| < 2^x, so that |scale * G| < 2^14.
// `factor` bounds what the kernel multiplies into the upstream gradients (an importance weight).
__device__ __forceinline__ void grad_scale(const float *upstream, long long T, float factor, FusedScalars *out) {
  __shared__ float red[kScaleFloats];
  float m = 0.f;
  for (long long t = threadIdx.x; t < T; t += blockDim.x) {
    const float v = fabsf(upstream[t]);
    if (v < __int_as_float(0x7f800000)) m = fmaxf(m, v);
  }
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < (int)(blockDim.x >> 5); ++w) m = fmaxf(m, red[w]);
    m *= factor;
    int x = 0;
    if (m > 0.f) frexpf(m, &x);
    int e = 14 - x;
    e = e > 60 ? 60 : (e < -60 ? -60 : e);
    out->scale = ldexpf(1.f, e);
    out->inv_scale = ldexpf(1.f, -e);
  }
}
__global__ void grad_scale_kernel(const float *upstream, long long T, float factor, FusedScalars *out) {
  begin_after(true);
  grad_scale(upstream, T, factor, out);
  if (threadIdx.x == 0) end_after(true);
}

// out[r, c] = float16(in[r, c]), in pieces of 8 elements, `per_row` of them in each of `rows` rows; kHalfPieces of them a
// block, four a thread.  Beside the first contraction's block an SM has room for one block with kBesidePair bytes of shared
// memory, and for 768 threads of 32 registers.  Short blocks: what is left when the contraction ends spreads over the whole chip (two blocks of
// 256 threads an SM that share all pieces: 88 us for 32,000 x 1,024, which the chip by itself copies in 22).
//
// The first block finds the scale of the upstream gradients.  (By a launch of its own in front of the contraction: 64 x 512 x
// 8,000 46.7 us a call, 45.0 this way, 1,200 x 1,024 x 16,000 200.8 / 198.6.)
constexpr int kHalfBlk = 768, kHalfPieces = 4 * kHalfBlk;
__global__ void __launch_bounds__(1024, 2)
to_half_kernel(const __nv_bfloat16 *in, long long ld_in, __half *out, long long ld_out, int rows, int per_row,
               const float *upstream, long long T, float factor, FusedScalars *scalars) {
  begin_after(true);
  if (blockIdx.x == 0) {
    grad_scale(upstream, T, factor, scalars);
    return;
  }
  const long long first = (blockIdx.x - 1LL) * kHalfPieces + threadIdx.x;
  const int r0 = (int)(first / per_row), c0 = (int)(first - (long long)r0 * per_row);
  const int dr = kHalfBlk / per_row, dc = kHalfBlk - dr * per_row;
  constexpr int kLoads = kHalfPieces / kHalfBlk;
  // f(step, row, piece of the row)
  const auto each = [&](auto f) {
    int r = r0, c = c0;
#pragma unroll
    for (int u = 0; u < kLoads; ++u) {
      if (r < rows) f(u, r, c);
      r += dr;
      c += dc;
      if (c >= per_row) {
        c -= per_row;
        ++r;
      }
    }
  };
  uint4 raw[kLoads];
  each([&](int u, int r, int c) { raw[u] = *reinterpret_cast<const uint4 *>(in + r * ld_in + c * 8); });
  each([&](int u, int r, int c) {
    const uint32_t b[4] = {raw[u].x, raw[u].y, raw[u].z, raw[u].w};
    uint32_t w[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const __half2 h = __floats2half2_rn(__uint_as_float(b[k] << 16), __uint_as_float(b[k] & 0xffff0000u));
      w[k] = *reinterpret_cast<const uint32_t *>(&h);
    }
    *reinterpret_cast<uint4 *>(out + r * ld_out + c * 8) = make_uint4(w[0], w[1], w[2], w[3]);
  });
  if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) end_after(true);  // the others leave their place to the next blocks
}

namespace {

size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

struct FusedLayout {
  long long Vp, Tp, panel;
  size_t off_scalars, off_lpt, off_lpi, off_fli, off_flt, off_wt, off_hs, off_z, off_g, off_rmax, off_rowscale,
      off_hidscale, off_acoef, total;
  long long max_pieces;
};

// The default panel: 4096 tokens, or as many as keep everything that it is made of within 1 GiB.  Every panel after the
// first adds to all of d_w (H = 2,864, V = 12,179: 98 us for 631 tokens, of which the products are 26).
constexpr long long kPanelRows = 4096, kPanelBytes = 1LL << 30;

bool fused_layout(const dvp_fused_args *a, FusedLayout *L, bool small = false) {
  if (a->T < 0 || a->H < 1 || a->V < 1) return false;
  L->Vp = (a->V + 15) / 16 * 16;
  L->max_pieces = (a->V + gemm::kBN - 1) / gemm::kBN;  // one per tile column of the logits contraction
  long long panel = a->panel_rows;
  if (panel == 0) {
    // logits and gradients, hidden rows, row maxima, three factors: what is taken by the panel's tokens below
    long long most = kPanelBytes / (6 * L->Vp + 2 * a->H + 4 * L->max_pieces + 12) / 128 * 128;
    if (most < kPanelRows || small) most = kPanelRows;
    panel = (a->T + 127) / 128 * 128;
    if (panel > most) panel = most;
    if (panel < 128) panel = 128;
  }
  if (panel % 128 != 0 || panel < 128) return false;
  L->panel = panel;
  L->Tp = (a->T + 7) / 8 * 8;
  if (L->Tp == 0) L->Tp = 8;
  size_t o = 0;
  auto take = [&](size_t bytes) {
    const size_t at = o;
    o = align_up(o + bytes, 256);
    return at;
  };
  L->off_scalars = take(sizeof(FusedScalars));
  L->off_lpt = take((size_t)a->T * 4);
  L->off_lpi = take((size_t)a->T * 4);
  L->off_fli = take((size_t)a->T);
  L->off_flt = take((size_t)a->T);
  L->off_wt = take((size_t)a->H * L->Vp * 2);
  L->off_hs = take((size_t)a->H * panel * 2);  // the panel's hidden rows, scaled, transposed, float16
  L->off_z = take((size_t)panel * L->Vp * 4);
  L->off_g = take((size_t)panel * L->Vp * 2);
  L->off_rmax = take((size_t)panel * L->max_pieces * 4);
  L->off_rowscale = take((size_t)panel * 4);
  L->off_hidscale = take((size_t)panel * 4);
  L->off_acoef = take((size_t)panel * 4);
  L->total = o;
  return true;
}

template <typename Kernel>
cudaError_t launch_both(Kernel kernel, size_t smem, const panel::PanelParams &pp, const RowParams &infer, cudaStream_t s) {
  if (smem > 48 * 1024) {
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
  }
  return launch_after(kernel, (unsigned)(infer.T + pp.row.T), panel::kSums / 2, smem, s, pp, infer);
}

dvp_side_out offset_side(const dvp_side_out &o, long long r0, long long words) {
  dvp_side_out r = o;
  if (r.max) r.max += r0;
  if (r.lse) r.lse += r0;
  if (r.lse_safe) r.lse_safe += r0;
  if (r.logp) r.logp += r0;
  if (r.logp_mp) r.logp_mp += r0;
  if (r.comp_mp) r.comp_mp += r0;
  if (r.count) r.count += r0;
  if (r.log_cov) r.log_cov += r0;
  if (r.mask) r.mask += r0 * words;
  return r;
}

}  // namespace
}  // namespace dvp

extern "C" {

size_t dvp_workspace_bytes(int entry_point, const void *args) {
  if (entry_point != DVP_ENTRY_FUSED_LMHEAD || !args) return 0;
  const dvp_fused_args *a = static_cast<const dvp_fused_args *>(args);
  if (a->struct_size != sizeof(dvp_fused_args)) return 0;
  dvp::FusedLayout L;
  return dvp::fused_layout(a, &L) ? L.total : 0;
}

int dvp_gemm_tn(const void *a, int64_t lda, const void *b, int64_t ldb, float *c, int64_t ldc, int64_t m,
                int64_t n, int64_t k, int32_t dtype, float alpha, int32_t accumulate, int32_t *status,
                void *stream) {
  if (!a || !b || !c || !status || m < 0 || n < 0 || k < 0) return DVP_ERR_INVALID_ARG;
  if (m > 0x7fffffffLL || n > 0x7fffffffLL || k > 0x7fffffffLL) return DVP_ERR_UNSUPPORTED;
  if (dtype != DVP_BF16 && dtype != DVP_F16) return DVP_ERR_UNSUPPORTED;
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return DVP_ERR_CUDA;
  const cudaError_t e =
      dvp::gemm::launch_gemm_tn(a, lda, b, ldb, c, ldc, (int)m, (int)n, (int)k, dtype == DVP_BF16, alpha,
                                nullptr, (accumulate & 1) != 0, status, sms,
                                static_cast<cudaStream_t>(stream), (accumulate & 2) != 0, (accumulate & 4) != 0,
                                (accumulate & 8) ? 2 : 1, nullptr, 0, nullptr, 0, dvp::gemm::Order::kAlone, 0,
                                (accumulate & 16) != 0);
  if (e == cudaErrorInvalidValue) return DVP_ERR_UNSUPPORTED;
  return e == cudaSuccess ? DVP_OK : DVP_ERR_CUDA;
}

int dvp_fused_lmhead_forward_backward(const dvp_fused_args *a) {
  using namespace dvp;
  if (!a || a->struct_size != sizeof(dvp_fused_args)) return DVP_ERR_INVALID_ARG;
  if (a->id_dtype != DVP_ID_I64 && a->id_dtype != DVP_ID_I32) return DVP_ERR_UNSUPPORTED;
  if (a->T < 0 || a->T > 0x7fffffffLL || a->H < 1 || a->V < 1) return DVP_ERR_INVALID_ARG;
  if (a->V > 0x7fffff00LL || a->H > 0x7fffff00LL) return DVP_ERR_UNSUPPORTED;
  if (!(a->rho >= 0.0 && a->rho <= 1.0)) return DVP_ERR_INVALID_ARG;
  FusedLayout L;
  if (!fused_layout(a, &L)) return DVP_ERR_INVALID_ARG;
  if (a->T == 0) return DVP_OK;
  if (!a->hidden || !a->w_vocab || !a->ids || !a->upstream || !a->d_hidden || !a->d_w)
    return DVP_ERR_INVALID_ARG;
  if (a->ld_hidden < a->H || a->ld_w < a->H || a->ld_dh < a->H || a->ld_dw < a->H)
    return DVP_ERR_INVALID_ARG;
  if (a->infer_logits && a->ld_infer < a->V) return DVP_ERR_INVALID_ARG;
  if (!a->infer_logits && a->log_ratio) return DVP_ERR_INVALID_ARG;
  if (a->weight_kind != DVP_WEIGHT_NONE) {
    if (a->weight_kind != DVP_WEIGHT_TRUNCATE && a->weight_kind != DVP_WEIGHT_MASK) return DVP_ERR_INVALID_ARG;
    if (!a->infer_logits) return DVP_ERR_INVALID_ARG;
    if (!(a->weight_lo >= 0.f && a->weight_hi >= a->weight_lo) || !std::isfinite(a->weight_hi))
      return DVP_ERR_INVALID_ARG;
  } else if (a->weight_out) {
    return DVP_ERR_INVALID_ARG;
  }
  if (a->ld_hidden % 8 || a->ld_w % 8 || a->ld_dh % 8 || a->ld_dw % 8 ||
      (uintptr_t)a->hidden % 16 || (uintptr_t)a->w_vocab % 16 || (uintptr_t)a->d_hidden % 32 ||
      (uintptr_t)a->d_w % 32)
    return DVP_ERR_UNSUPPORTED;
  // a workspace for panels of 4096 tokens is enough for the default
  if (a->panel_rows == 0 && a->workspace_bytes < L.total) (void)fused_layout(a, &L, true);
  if (!a->workspace || (uintptr_t)a->workspace % 256 || a->workspace_bytes < L.total)
    return DVP_ERR_WORKSPACE;

  cudaStream_t s = static_cast<cudaStream_t>(a->stream);
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return DVP_ERR_CUDA;

  char *ws = static_cast<char *>(a->workspace);
  FusedScalars *sc = reinterpret_cast<FusedScalars *>(ws + L.off_scalars);
  float *lpt = a->train.logp_mp ? a->train.logp_mp : reinterpret_cast<float *>(ws + L.off_lpt);
  float *lpi = a->infer.logp_mp ? a->infer.logp_mp : reinterpret_cast<float *>(ws + L.off_lpi);
  uint8_t *fli = reinterpret_cast<uint8_t *>(ws + L.off_fli);
  uint8_t *flt = a->flags ? a->flags : reinterpret_cast<uint8_t *>(ws + L.off_flt);
  __half *w16 = reinterpret_cast<__half *>(ws + L.off_wt);    // W in float16: [V, H] as it lies, or [H, Vp]
  __half *hs16 = reinterpret_cast<__half *>(ws + L.off_hs);   // [H, panel]: the panel's hidden rows, scaled, transposed
  float *z = reinterpret_cast<float *>(ws + L.off_z);         // [panel, Vp] logits
  __half *p16 = reinterpret_cast<__half *>(ws + L.off_g);     // [panel, Vp] P = 2^14 e^{z - m} on the safe set
  float *rmax = reinterpret_cast<float *>(ws + L.off_rmax);   // [panel, max_pieces] row maxima of z in pieces
  float *row_scale = reinterpret_cast<float *>(ws + L.off_rowscale);  // [panel] factor of each row of P
  float *hid_scale = reinterpret_cast<float *>(ws + L.off_hidscale);  // [panel] the same times a power of two
  float *a_coef = reinterpret_cast<float *>(ws + L.off_acoef);        // [panel] coefficient of the 1[k = a] term
  const __nv_bfloat16 *hidden = static_cast<const __nv_bfloat16 *>(a->hidden);
  const __nv_bfloat16 *w = static_cast<const __nv_bfloat16 *>(a->w_vocab);
  const int T = (int)a->T, H = (int)a->H, V = (int)a->V;
  const long long id_bytes = a->id_dtype == DVP_ID_I32 ? 4 : 8;
  const long long mask_words = (a->V + 31) / 32;

  const bool weighted = a->weight_kind != DVP_WEIGHT_NONE;
  const float factor = weighted ? fmaxf(1.f, a->weight_hi) : 1.f;

  const double log_rho = a->rho > 0.0 ? std::log(a->rho) : -HUGE_VAL;
  // the inference rows: a forward-only row pass over the stored logits
  RowParams infer{};
  if (a->infer_logits) {
    RowParams &p = infer;
    p.train = a->infer_logits;
    p.ids = a->ids;
    p.T = a->T;
    p.V = a->V;
    p.ld_train = a->ld_infer;
    p.log_rho = log_rho;
    p.id_is_i32 = a->id_dtype == DVP_ID_I32;
    p.out_t = a->infer;
    p.out_t.logp_mp = lpi;
    p.flags = fli;
    p.bounds_status = bounds_status_word();
  }
  const two_sweeps::Shape infer_shape = a->infer_logits ? two_sweeps::shape_of(infer) : two_sweeps::Shape{};
  // ... in one launch with the panel's rows (dvp_both_rows_kernel), where four blocks of both fit an SM
  const bool both = a->infer_logits && !weighted && a->T <= L.panel && infer_shape.smem <= 55 * 1024 &&
                    (infer_shape.threads == panel::kSums / 2 || infer_shape.threads == 0);
  // W as d_hidden's contraction reads it: as it lies, [V, H], the transposed (MN-major) B operand; transposed where H is not a
  // multiple of 8, the unit of TMA's strides.
  const bool w_lies = H % 8 == 0;
  const long long ld_w16 = w_lies ? H : L.Vp;
  int panel_index = 0;
  for (long long r0 = 0; r0 < a->T; r0 += L.panel, ++panel_index) {
    const int rows = (int)((a->T - r0 < L.panel) ? a->T - r0 : L.panel);
    // logits of the panel: z = hidden[r0 : r0 + rows] x W^T (bf16 operands, fp32 accumulate)
    // its epilogue also leaves each row's maximum, one piece per tile column: the panel's row pass
    // then knows the threshold before it reads the panel.  Early from the second panel on: the launch before it is
    // the last of d_w's, when nobody reads z or the maxima any more
    cudaError_t e = gemm::launch_gemm_tn(hidden + r0 * a->ld_hidden, a->ld_hidden, w, a->ld_w, z, L.Vp,
                                         rows, V, H, true, 1.f, nullptr, false, &sc->status, sms, s, false,
                                         false, 1, rmax, L.max_pieces, nullptr, 0,
                                         panel_index == 0 ? gemm::Order::kFirst : gemm::Order::kEarly);
    if (e != cudaSuccess) return e == cudaErrorInvalidValue ? DVP_ERR_UNSUPPORTED : DVP_ERR_CUDA;
    if (panel_index == 0) {
      // While the first contraction runs: the inference rows, where they have a launch of their own (the panel's rows take
      // the log-ratio and the importance weight from them), on SMs that it does not use or has left, since their blocks
      // take more shared memory than kBesidePair; behind them W, whose blocks lie beside the contraction's.
      if (a->infer_logits && !both && two_sweeps::launch(infer, s) != cudaSuccess) return DVP_ERR_CUDA;
      if (w_lies) {
        (void)launch_after(to_half_kernel, (unsigned)(((long long)V * (H / 8) + kHalfPieces - 1) / kHalfPieces + 1), kHalfBlk, 0,
                           s, w, a->ld_w, w16, ld_w16, V, H / 8, a->upstream, a->T, factor, sc);
      } else {
        (void)launch_after(grad_scale_kernel, 1, 1024, 0, s, a->upstream, a->T, factor, sc);
        launch_transpose<__nv_bfloat16, __half>(w, a->ld_w, w16, ld_w16, V, H, s);
      }
      if (cudaGetLastError() != cudaSuccess) return DVP_ERR_CUDA;
    }
    // rows of the panel, one sweep: statistics, and the gradient panel up to a factor per row
    panel::PanelParams pp{};
    RowParams &p = pp.row;
    p.train = z;
    p.ids = static_cast<const char *>(a->ids) + r0 * id_bytes;
    p.upstream = a->upstream + r0;
    p.T = rows;
    p.V = a->V;
    p.ld_train = L.Vp;
    p.log_rho = log_rho;
    p.id_is_i32 = a->id_dtype == DVP_ID_I32;
    p.out_t = offset_side(a->train, r0, mask_words);
    p.out_t.logp_mp = lpt + r0;
    p.flags = flt + r0;
    p.bounds_status = bounds_status_word();
    panel::MeetParams meet{};
    if (both) {
      meet = {lpt, lpi, flt, fli, a->log_ratio};
    } else if (a->infer_logits) {
      pp.logp_mp_i = lpi + r0;
      pp.flags_i = fli + r0;
      p.log_ratio = a->log_ratio ? a->log_ratio + r0 : nullptr;
    }
    if (weighted) {
      p.weight_kind = (int)a->weight_kind;
      p.weight_lo = a->weight_lo;
      p.weight_hi = a->weight_hi;
      p.weight_out = a->weight_out ? a->weight_out + r0 : nullptr;
    }
    pp.row_max = rmax;
    pp.row_max_ld = L.max_pieces;
    pp.row_max_n = (int)L.max_pieces;
    pp.P = p16;
    pp.ld_p = L.Vp;
    pp.row_scale = row_scale;
    pp.hid_scale = hid_scale;
    pp.a_coef = a_coef;
    pp.scale = &sc->scale;
    // Few rows: as many threads a row as it has sums.  More than fill the chip: half of them, so that one row's reductions
    // and results pass beside the sweeps of three others.  us a call with the first form / the second: 163 x 416 x 45,277
    // 138 / 146, 767 x 1,448 x 10,474 172 / 170, 4,727 x 2,864 x 12,179 1,274 / 1,224, 3,891 x 2,752 x 58,933 4,220 / 3,997.
    const cudaError_t pe = both && infer_shape.threads
                               ? launch_both(panel::dvp_both_rows_kernel<false>, infer_shape.smem, pp, infer, s)
                           : both ? launch_both(panel::dvp_both_rows_kernel<true>, infer_shape.smem, pp, infer, s)
                           : rows < 4 * 148
                               ? launch_after(panel::dvp_panel_kernel<1, 4>, (unsigned)rows, panel::kSums, 0, s, pp)
                               : launch_after(panel::dvp_panel_kernel<2, 1>, (unsigned)rows, panel::kSums / 2, 0, s, pp);
    if (pe != cudaSuccess) return DVP_ERR_CUDA;
    // d_hidden[r0 : r0 + rows] = diag(c) P W + q_t W[a_t]: the factor is applied per row and the 1[k = a] term
    // added in fp32.  Few output tiles and a long K: each tile is computed as several K ranges, whose partial
    // results go where the logits were (read for the last time by the row pass) and are summed in order.
    const long long dh_tiles = ((rows + 255) / 256) * (long long)((H + 255) / 256), Hp = (H + 7) / 8 * 8;
    const int room = (int)(L.panel * L.Vp / ((long long)rows * Hp) < 32 ? L.panel * L.Vp / ((long long)rows * Hp) : 32);
    const int ranges = gemm::choose_ranges(dh_tiles, V, sms / 2, room > 1 ? room : 1, (double)rows * Hp * 4);
    float *dh = a->d_hidden + r0 * a->ld_dh;
    e = ranges > 1 ? gemm::launch_gemm_tn(p16, L.Vp, w16, ld_w16, z, Hp, rows, H, V, false, 1.f, nullptr, false,
                                          &sc->status, sms, s, false, false, ranges, nullptr, 0, nullptr, rows * Hp,
                                          gemm::Order::kAfter, 0, w_lies)
                   : gemm::launch_gemm_tn(p16, L.Vp, w16, ld_w16, dh, a->ld_dh, rows, H, V, false, 1.f, nullptr, false,
                                          &sc->status, sms, s, false, false, 1, nullptr, 0, row_scale, 0,
                                          gemm::Order::kAfter, 0, w_lies);
    // while it runs, on SMs that it does not use or has left: the panel's hidden rows times their factor (and
    // 2^14 * scale / 512), transposed, in float16
    launch_transpose<__nv_bfloat16, __half>(hidden + r0 * a->ld_hidden, a->ld_hidden, hs16, L.panel, rows, H, s,
                                            hid_scale);
    if (e == cudaSuccess)
      e = launch_after(panel::sum_ranges_kernel, (unsigned)(((H + 1023) / 1024) * (long long)rows), 256, 0, s,
                       ranges > 1 ? z : dh, rows * Hp, ranges > 1 ? Hp : a->ld_dh, ranges,
                       ranges > 1 ? row_scale : nullptr, dh, a->ld_dh, w, a->ld_w, p.ids, p.id_is_i32, a_coef, H, meet);
    if (e != cudaSuccess) return e == cudaErrorInvalidValue ? DVP_ERR_UNSUPPORTED : DVP_ERR_CUDA;
    // d_w (+)= P^T x (scaled hidden rows) * 512 / (2^14 scale): P is read as it lies, [rows, V] with V
    // contiguous, as the transposed (MN-major) A operand of the contraction; it needs nothing of sum_ranges_kernel
    e = gemm::launch_gemm_tn(p16, L.Vp, hs16, L.panel, a->d_w, a->ld_dw, V, H, rows, false, 1.f / 32.f,
                             &sc->inv_scale, panel_index > 0 || a->accumulate_dw != 0, &sc->status, sms,
                             s, false, true, 1, nullptr, 0, nullptr, 0, gemm::Order::kEarly, gemm::kChainK);
    if (e != cudaSuccess) return e == cudaErrorInvalidValue ? DVP_ERR_UNSUPPORTED : DVP_ERR_CUDA;
    // ... + q_t hidden_t into row a_t of d_w: tokens that share a row are added in token order
    for (int c0 = 0; c0 < rows; c0 += panel::kIdChunk) {
      const int n = rows - c0 < panel::kIdChunk ? rows - c0 : panel::kIdChunk;
      const void *ids_c = static_cast<const char *>(p.ids) + (long long)c0 * id_bytes;
      (void)launch_after(panel::add_sampled_hidden_kernel, (unsigned)((n + panel::kSampledWarps - 1) / panel::kSampledWarps),
                         panel::kSampledWarps * 32, panel::kSampledSmem, s, ids_c, p.id_is_i32, a_coef + c0, n,
                         hidden + (r0 + c0) * a->ld_hidden, a->ld_hidden, a->d_w, a->ld_dw, H);
    }
    if (cudaGetLastError() != cudaSuccess) return DVP_ERR_CUDA;
  }

  return cudaGetLastError() == cudaSuccess ? DVP_OK : DVP_ERR_CUDA;
}


// ---- a variant that allocates nothing ------------------------------------------
// The workspace of the fused entry point, taken from a fixed array that is part
// of the loaded library instead of from the caller.  In host code the array's
// name is only a handle; the device address comes from cudaGetSymbolAddress, once
// per device, with that device current.

}  // extern "C"

namespace {
constexpr size_t kStaticWorkspaceBytes = (size_t)DVP_STATIC_WORKSPACE_BYTES;
static __device__ __align__(256) unsigned char g_static_workspace[kStaticWorkspaceBytes];
constexpr int kMaxDevices = 64;
void *g_static_workspace_ptr[kMaxDevices] = {};
std::mutex g_static_workspace_mutex;
}  // namespace

extern "C" {

int dvp_fused_lmhead_forward_backward_static(const dvp_fused_args *a) {
  if (!a || a->struct_size != sizeof(dvp_fused_args)) return DVP_ERR_INVALID_ARG;
  dvp_fused_args b = *a;
  if (b.panel_rows == 0) b.panel_rows = 128;  // the smallest panel leaves the most room
  dvp::FusedLayout L;
  if (!dvp::fused_layout(&b, &L)) return DVP_ERR_INVALID_ARG;
  if (L.total > kStaticWorkspaceBytes) return DVP_ERR_WORKSPACE;  // beyond the built-in maximum
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return DVP_ERR_CUDA;
  if (dev < 0 || dev >= kMaxDevices) return DVP_ERR_UNSUPPORTED;
  void *ptr = nullptr;
  {
    std::lock_guard<std::mutex> lock(g_static_workspace_mutex);
    if (!g_static_workspace_ptr[dev]) {
      void *sym = nullptr;
      if (cudaGetSymbolAddress(&sym, g_static_workspace) != cudaSuccess || !sym) return DVP_ERR_CUDA;
      g_static_workspace_ptr[dev] = sym;
    }
    ptr = g_static_workspace_ptr[dev];
  }
  b.workspace = ptr;
  b.workspace_bytes = kStaticWorkspaceBytes;
  return dvp_fused_lmhead_forward_backward(&b);
}

int dvp_static_workspace_status(uint32_t *status_out) {
  if (!status_out) return DVP_ERR_INVALID_ARG;
  if (cudaDeviceSynchronize() != cudaSuccess) return DVP_ERR_CUDA;
  // the status is the first word of the workspace, here of the built-in array
  return cudaMemcpyFromSymbol(status_out, g_static_workspace, sizeof(uint32_t)) == cudaSuccess ? DVP_OK
                                                                                              : DVP_ERR_CUDA;
}

}  // extern "C"
