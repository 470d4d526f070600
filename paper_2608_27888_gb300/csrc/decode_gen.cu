// Decoders of a general shape (Sec. 4's decoder and the A x B sizes of its
// MLP ablation): num_levels x channels latent features (4- or 8-channel
// grids) concatenated with a positional encoding of F frequencies, 1..4 hidden
// layers of width 16..128, ReLU or LeakyReLU, sigmoid output.
//
//   k_decode_gen_tc   bucketed 128-query tiles on the tensor-core pipeline of
//                     decode_pipe.cuh; the producers gather a row's latents
//                     (L levels of C channels, packed fp16 blend) and append
//                     the positional encoding.
//   k_decode_gen_fma  per-lane fp32 FMAs, one query per thread (the fp32
//                     precision's bucketed path, and every precision's
//                     divergent-FMA mode): the same rounding rules as the
//                     standard per-lane kernel.
#include <math.h>

#include "decode_pipe.cuh"

namespace ntc {
namespace {

__device__ __forceinline__ void count_bad_warp(bool bad, unsigned long long *err) {
  const unsigned m = __ballot_sync(0xFFFFFFFFu, bad);
  if (m && (threadIdx.x & 31) == __ffs(m) - 1) atomicAdd(err, (unsigned long long)__popc(m));
}

// How a general shape fills the pipeline: two converters, four slots up to
// H = 64 and two at H = 128, and four producer stages, or two where tensor
// memory holds no more.  Rows of 16 latent channels keep so many taps in
// registers that only two producer warpgroups fit.
template <int H, int LC>
struct GenShape {
  static constexpr int NE = 2, T = H == 128 ? 2 : 4, NP = LC <= 8 ? 4 : 2;
};
template <int H, bool BF16, int LC>
using GenPipe = Pipe<H, BF16, GenShape<H, LC>::NP, GenShape<H, LC>::NE, GenShape<H, LC>::T, 0, 0>;

// The producers: a thread builds one row of a tile.
template <int H, bool BF16, int L, int C>
__device__ __forceinline__ void produce_gen(const GenPipe<H, BF16, L * C> &pipe, const Assets &A, const Buckets &B,
                                            const GridDesc *grids, void *out, unsigned long long *err) {
  constexpr int NF = L * C + 4 * kGenMaxPe;  // feature values this input layout can have
  constexpr int LW = L * C / 2, NW = (NF + 15) / 16 * 8;
  const uint32_t K = pipe.K;
  constexpr uint32_t NP = GenShape<H, L * C>::NP;
  const uint32_t p = (uint32_t)pipe.warp >> 2, row = threadIdx.x & 127;  // tiles p, p + NP, ...
  typename GenPipe<H, BF16, L * C>::Rows rows(pipe, B, p);
  for (uint32_t k = p, j = 0; k < K && !pipe.wait.stopped(); k += NP, ++j) {
    const ntc_query q = rows.record();
    const uint32_t oi = rows.oi;
    const bool valid = oi != kNoRow;
    const bool good = valid && !query_bad(A, q);
    rows.look_ahead(pipe, k, rows.oi);
    const bool bad = valid && !good;
    count_bad_warp(bad, err);
    if (bad) put_nan_row(out, oi, pipe.P.out_dim, pipe.P.out_half);
    // the feature row, packed to fp16/bf16 pairs as it is produced: the latent
    // features, then sin/cos pairs of the encoding (zeros beyond)
    uint32_t pk[NW];
#pragma unroll
    for (int i = 0; i < NW; ++i) pk[i] = 0u;
    if (good) {
      {
        __half2 hl[LW];
        gen_latents_h2<L, C>(A, grids, q, hl);
#pragma unroll
        for (int i = 0; i < LW; ++i) {
          if (BF16) {
            const float2 x = __half22float2(hl[i]);
            pk[i] = pack<true>(x.x, x.y);
          } else {
            pk[i] = *reinterpret_cast<const uint32_t *>(&hl[i]);
          }
        }
      }
      const uint32_t F = A.pe_frequencies;
      if (F) {
        // sin/cos(2 pi u) from the hardware approximation, after reducing u
        // to [-1/2, 1/2] (exact), where its absolute error is about 2^-21:
        // far below the fp16/bf16 rounding the features then go through
        float u, v, su, cu, sv, cv;
        pe_coords(A, q, u, v);
        __sincosf(6.28318530718f * __fsub_rn(u, rintf(u)), &su, &cu);
        __sincosf(6.28318530718f * __fsub_rn(v, rintf(v)), &sv, &cv);
#pragma unroll
        for (int f = 0; f < kGenMaxPe; ++f) {
          if (LW + 2 * f + 1 >= NW) break;
          if (f < (int)F) {
            pk[LW + 2 * f] = pack<BF16>(su, cu);
            pk[LW + 2 * f + 1] = pack<BF16>(sv, cv);
            const float su2 = 2.0f * su * cu, cu2 = cu * cu - su * su;
            const float sv2 = 2.0f * sv * cv, cv2 = cv * cv - sv * sv;
            su = su2, cu = cu2, sv = sv2, cv = cv2;
          }
        }
      }
    }
    if (k < pipe.Kg) pipe.hand_over(p, j, k, row, pk, good ? oi : kNoRow);  // (a bad bucket's rows end here)
  }
}

template <int H, bool BF16, int L, int C>
__global__ void __launch_bounds__(GenPipe<H, BF16, L * C>::kThreads, 1)
    k_decode_gen_tc(Assets A, Buckets B, const __grid_constant__ PipeArgs P, void *out, unsigned long long *err,
                    unsigned int *status) {
  extern __shared__ __align__(128) uint8_t smem[];
  const GridDesc *grids = A.grids;
  const GenPipe<H, BF16, L * C> pipe(P, smem, B, A.num_decoders, status, grids, A.num_sets * L * A.num_mips);
  if (pipe.warp < pipe.kWarpE)
    produce_gen<H, BF16, L, C>(pipe, A, B, grids, out, err);
  else
    pipe.consume(out);
  pipe.end();
}

template <typename T>
struct Op;
template <>
struct Op<float> {
  static __device__ __forceinline__ float ld(const float *p) { return __ldg(p); }
  static __device__ __forceinline__ float round(float x) { return x; }
  static __device__ __forceinline__ float cvt(float x) { return x; }
};
template <>
struct Op<__half> {
  static __device__ __forceinline__ float ld(const __half *p) { return __half2float(__ldg(p)); }
  static __device__ __forceinline__ float round(float x) { return __half2float(__float2half_rn(x)); }
  static __device__ __forceinline__ __half cvt(float x) { return __float2half_rn(x); }
};
template <>
struct Op<__nv_bfloat16> {
  static __device__ __forceinline__ float ld(const __nv_bfloat16 *p) { return __bfloat162float(__ldg(p)); }
  static __device__ __forceinline__ float round(float x) { return __bfloat162float(__float2bfloat16_rn(x)); }
  static __device__ __forceinline__ __nv_bfloat16 cvt(float x) { return __float2bfloat16_rn(x); }
};

__device__ __forceinline__ float act_f(float x, uint32_t act, float slope) {
  return x > 0.0f ? x : (act == 1 ? slope * x : 0.0f);
}

// Per-lane decode of a general shape; row i is row i of the bucketed order B
// (bucketed != 0) or query i of qs itself, written to its output row.
template <typename T>
__global__ void __launch_bounds__(128) k_decode_gen_fma(Assets A, GenWeights G, const ntc_query *qs, int bucketed,
                                                        Buckets B, size_t n, float *out, unsigned long long *err) {
  const bool copied = bucketed && rows_copied(B, A.num_decoders);
  using E = Op<T>;
  const uint32_t H = G.hidden, I = G.in_dim, C = G.out_dim, NL = G.layers, CP = out_pad(C);
  const size_t wbytes = (((size_t)H * I + (size_t)(NL - 1) * H * H + (size_t)H * CP) * sizeof(T) + 15) / 16 * 16;
  const size_t step = (size_t)gridDim.x * blockDim.x;
  const size_t nr = (n + 31) & ~(size_t)31;  // whole warps iterate together
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < nr; i += step) {
    const bool valid = i < n;
    ntc_query q;
    uint32_t oi = 0;
    bool bad = false;
    if (valid) {
      if (bucketed) {
        bucket_row(B, copied, (uint32_t)i, oi, q);
      } else {
        q = load_query(qs + i);
        oi = (uint32_t)i;
      }
      bad = query_bad(A, q);
    }
    count_bad_warp(valid && bad, err);
    if (!valid) continue;
    float *o_row = out + (size_t)oi * C;
    if (bad) {
      for (uint32_t c = 0; c < C; ++c) o_row[c] = __int_as_float(0x7fc00000);
      continue;
    }
    const uint8_t *img = G.fma + (size_t)__ldg(A.map + q.set_id) * G.fma_stride;
    const T *W = reinterpret_cast<const T *>(img);
    const float *bias = reinterpret_cast<const float *>(img + wbytes);
    float f[kGenMaxIn];
    gen_features(A, A.grids, q, f);
    float h[kGenMaxHidden], g[kGenMaxHidden];
    for (uint32_t j = 0; j < H; ++j) {
      float acc = 0.0f;
      for (uint32_t k = 0; k < I; ++k) acc = fmaf(E::ld(W + (size_t)j * I + k), E::round(f[k]), acc);
      h[j] = E::round(act_f(acc + __ldg(bias + j), G.activation, G.slope));
    }
    const T *Wl = W + (size_t)H * I;
    for (uint32_t l = 1; l < NL; ++l) {
      for (uint32_t j = 0; j < H; ++j) {
        float acc = 0.0f;
        for (uint32_t k = 0; k < H; ++k) acc = fmaf(E::ld(Wl + (size_t)j * H + k), h[k], acc);
        g[j] = E::round(act_f(acc + __ldg(bias + l * H + j), G.activation, G.slope));
      }
      for (uint32_t j = 0; j < H; ++j) h[j] = g[j];
      Wl += (size_t)H * H;
    }
    const T *Wo = Wl;  // W_out^T [H][CP]
    for (uint32_t c = 0; c < C; ++c) {
      float acc = 0.0f;
      for (uint32_t j = 0; j < H; ++j) acc = fmaf(E::ld(Wo + (size_t)j * CP + c), h[j], acc);
      o_row[c] = 1.0f / (1.0f + expf(-(acc + __ldg(bias + NL * H + c))));
    }
  }
}

// One CTA per decoder: fp32 weights (W1, b1, {W_l, b_l}..., Wout, bout) ->
// the tcgen05 image (if tc) and the per-lane image of type T.
template <typename T>
__global__ void k_pack_gen(const float *w32, GenWeights G, uint8_t *tc, uint8_t *fma) {
  using E = Op<T>;
  const uint32_t d = blockIdx.x, H = G.hidden, I = G.in_dim, C = G.out_dim, NL = G.layers, K1 = G.k1;
  const uint32_t CP = out_pad(C);
  const size_t P = (size_t)H * I + H + (size_t)(NL - 1) * (H * H + H) + (size_t)C * H + C;
  const float *p = w32 + (size_t)d * P;
  // source offsets of each layer
  auto Wsrc = [&](uint32_t l) -> const float * {  // l = 0: W1; 1..NL-1: hidden; NL: output
    return l == 0 ? p : p + (size_t)H * I + H + (size_t)(l - 1) * (H * H + H);
  };
  auto bsrc = [&](uint32_t l) -> const float * {
    return l == 0 ? p + (size_t)H * I : Wsrc(l) + (size_t)(l < NL ? H : C) * H;
  };
  if (tc) {
    uint8_t *img = tc + (size_t)d * G.tc_stride;
    uint8_t *base = img;
    for (uint32_t l = 0; l <= NL; ++l) {  // [rows][K + 16]: the weights, then the bias parts
      const uint32_t rows = l < NL ? H : 16, real = l < NL ? H : C, in = l ? H : I, K = (l ? H : K1) + 16;
      for (uint32_t e = threadIdx.x; e < rows * K; e += blockDim.x) {
        const uint32_t r = e / K, k = e % K;
        T v = T(0.0f);
        if (r < real && k < in) v = E::cvt(Wsrc(l)[(size_t)r * in + k]);
        else if (r < real && k >= K - 16 && k < K - 16 + kBiasParts) v = bias_part<T>(bsrc(l)[r], k - (K - 16));
        *reinterpret_cast<T *>(base + core_off(r, k, K)) = v;
      }
      base += (size_t)rows * K * 2;
    }
  }
  T *o = reinterpret_cast<T *>(fma + (size_t)d * G.fma_stride);
  for (uint32_t e = threadIdx.x; e < H * I; e += blockDim.x) o[e] = E::cvt(Wsrc(0)[e]);
  T *ol = o + (size_t)H * I;
  for (uint32_t l = 1; l < NL; ++l, ol += (size_t)H * H)
    for (uint32_t e = threadIdx.x; e < H * H; e += blockDim.x) ol[e] = E::cvt(Wsrc(l)[e]);
  for (uint32_t e = threadIdx.x; e < H * CP; e += blockDim.x) {
    const uint32_t j = e / CP, c = e % CP;
    ol[e] = E::cvt(c < C ? Wsrc(NL)[(size_t)c * H + j] : 0.0f);
  }
  const size_t wbytes = (((size_t)H * I + (size_t)(NL - 1) * H * H + (size_t)H * CP) * sizeof(T) + 15) / 16 * 16;
  float *ob = reinterpret_cast<float *>(fma + (size_t)d * G.fma_stride + wbytes);
  for (uint32_t e = threadIdx.x; e < NL * H + CP; e += blockDim.x) {
    const uint32_t l = e / H;
    ob[e] = l < NL ? bsrc(l)[e % H] : (e - NL * H < C ? bsrc(NL)[e - NL * H] : 0.0f);
  }
}

template <int H, bool BF16, int L, int C>
cudaError_t launch_gen_tc_t(const Assets &A, const GenWeights &G, const Buckets &B, size_t n, void *out,
                            unsigned long long *err, unsigned int *status, int num_sms, cudaStream_t st) {
  using S = GenShape<H, L * C>;
  using Pp = GenPipe<H, BF16, L * C>;
  constexpr uint32_t kMostSmem = 232448;  // dynamic shared memory of one CTA
  const uint32_t ngrids = A.num_sets * L * A.num_mips;
  const uint32_t stages = pipe_columns(H, S::T, G.k1, S::NP) <= 512 ? S::NP : 2;
  static_assert(pipe_columns(H, S::T, kGenMaxIn - 16, 2) <= 512, "tensor memory plan exceeds 512 columns");
  if (pipe_columns(H, S::T, G.k1, stages) > 512) return cudaErrorInvalidConfiguration;
  // images in shared memory: four, one per slot or more, so that the next
  // decoder's weights arrive early; at H = 128, where any number works (Pipe), as
  // many as fit (four hidden layers: one)
  uint32_t ns = 4;
  static_assert(H == 128 || S::T <= 4, "an image per slot");
  auto args = [&]() {
    return pipe_args(G.tc, G.tc_stride, G.k1, H, G.layers, ns, S::NP, stages, ngrids, A.num_decoders, G.out_dim, G.out_half, out, n);
  };
  PipeArgs P = args();
  while (H == 128 && ns > 1 && P.sm.total > kMostSmem) {
    --ns;
    P = args();
  }
  if (P.sm.total > kMostSmem) return cudaErrorInvalidConfiguration;
  P.act = G.activation == 1 && G.slope >= 0.0f && G.slope <= 1.0f ? 2u : G.activation;
  P.slope = G.slope;
  const uint32_t h = BF16 ? __bfloat16_as_ushort(__float2bfloat16_rn(G.slope)) : __half_as_ushort(__float2half_rn(G.slope));
  P.slope2 = h | h << 16;
  const auto kernel = k_decode_gen_tc<H, BF16, L, C>;
  static PerDevice attr;
  cudaError_t e = attr.once([&]() { return allow_smem((const void *)kernel, kMostSmem); });
  if (e != cudaSuccess) return e;
  const size_t max_tiles = (n + kTile - 1) / kTile + A.num_decoders + 1;
  size_t grid = (size_t)num_sms;
  if (grid > max_tiles) grid = max_tiles;
  e = launch_pdl_l1(kernel, dim3((unsigned)grid), dim3(Pp::kThreads), P.sm.total, st, A, B, P, out, err, status);
  if (e != cudaSuccess) return e;
  return cudaGetLastError();
}

template <int H, bool BF16>
cudaError_t launch_gen_tc_h(const Assets &A, const GenWeights &G, const Buckets &B, size_t n, void *out,
                            unsigned long long *err, unsigned int *status, int num_sms, cudaStream_t st) {
  if (A.channels == 8)
    return A.num_levels == 2 ? launch_gen_tc_t<H, BF16, 2, 8>(A, G, B, n, out, err, status, num_sms, st)
                             : launch_gen_tc_t<H, BF16, 1, 8>(A, G, B, n, out, err, status, num_sms, st);
  return A.num_levels == 2 ? launch_gen_tc_t<H, BF16, 2, 4>(A, G, B, n, out, err, status, num_sms, st)
                           : launch_gen_tc_t<H, BF16, 1, 4>(A, G, B, n, out, err, status, num_sms, st);
}

template <bool BF16>
cudaError_t launch_gen_tc_b(const Assets &A, const GenWeights &G, const Buckets &B, size_t n, void *out,
                            unsigned long long *err, unsigned int *status, int num_sms, cudaStream_t st) {
  if (G.hidden == 16) return launch_gen_tc_h<16, BF16>(A, G, B, n, out, err, status, num_sms, st);
  if (G.hidden == 32) return launch_gen_tc_h<32, BF16>(A, G, B, n, out, err, status, num_sms, st);
  if (G.hidden == 64) return launch_gen_tc_h<64, BF16>(A, G, B, n, out, err, status, num_sms, st);
  return launch_gen_tc_h<128, BF16>(A, G, B, n, out, err, status, num_sms, st);
}

template <typename T>
cudaError_t launch_gen_fma_t(const Assets &A, const GenWeights &G, const Buckets *B, const ntc_query *q, size_t n,
                             float *out, unsigned long long *err, int num_sms, cudaStream_t st) {
  int occ = 1;
  occ = resident_ctas(k_decode_gen_fma<T>, 128, 0);
  if (occ < 1) occ = 1;
  const size_t blocks = (n + 127) / 128;
  size_t grid = (size_t)num_sms * occ * 4;
  if (grid > blocks) grid = blocks;
  k_decode_gen_fma<T><<<(unsigned)grid, 128, 0, st>>>(A, G, q, B ? 1 : 0, B ? *B : Buckets{}, n, out, err);
  return cudaGetLastError();
}

}  // namespace

size_t gen_tc_image_bytes(uint32_t in_dim, uint32_t H, uint32_t layers) {
  return pipe_image_bytes(gen_k1(in_dim), H, layers);
}

cudaError_t launch_decode_gen_tc(const Assets &A, const GenWeights &G, const Buckets &B, size_t n, void *out,
                                 unsigned long long *err, unsigned int *status, bool bf16, int num_sms,
                                 cudaStream_t st, int *launches) {
  *launches += 1;
  return bf16 ? launch_gen_tc_b<true>(A, G, B, n, out, err, status, num_sms, st)
              : launch_gen_tc_b<false>(A, G, B, n, out, err, status, num_sms, st);
}

cudaError_t launch_decode_gen_fma(const Assets &A, const GenWeights &G, const Buckets *B, const ntc_query *q,
                                  size_t n, float *out, unsigned long long *err, ntc_precision prec, int num_sms,
                                  cudaStream_t st, int *launches) {
  *launches += 1;
  if (prec == NTC_PREC_FP32) return launch_gen_fma_t<float>(A, G, B, q, n, out, err, num_sms, st);
  if (prec == NTC_PREC_TC_BF16) return launch_gen_fma_t<__nv_bfloat16>(A, G, B, q, n, out, err, num_sms, st);
  return launch_gen_fma_t<__half>(A, G, B, q, n, out, err, num_sms, st);
}

cudaError_t launch_pack_gen(const float *w32, uint32_t D, const GenWeights &G, ntc_precision prec, uint8_t *tc,
                            uint8_t *fma, cudaStream_t st) {
  if (prec == NTC_PREC_FP32)
    k_pack_gen<float><<<D, 256, 0, st>>>(w32, G, nullptr, fma);
  else if (prec == NTC_PREC_TC_BF16)
    k_pack_gen<__nv_bfloat16><<<D, 256, 0, st>>>(w32, G, tc, fma);
  else
    k_pack_gen<__half><<<D, 256, 0, st>>>(w32, G, tc, fma);
  return cudaGetLastError();
}

}  // namespace ntc
