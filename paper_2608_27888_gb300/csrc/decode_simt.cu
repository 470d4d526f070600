// CUDA-core kernels: the fp32 reference decode over bucketed tiles, the debug
// kernels (taps, features) and the packing of decoder weights into the images
// the tensor-core kernels read.
#include <math.h>

#include "ntc_internal.cuh"

namespace ntc {
namespace {

__device__ __forceinline__ void count_bad(bool bad, unsigned long long *err) {
  unsigned m = __ballot_sync(0xFFFFFFFFu, bad);
  if (m && (threadIdx.x & 31) == __ffs(m) - 1) atomicAdd(err, (unsigned long long)__popc(m));
}

// fp32 decode over bucketed tiles: a CTA multiplies a tile's 128 activation
// columns by its decoder's matrices out of shared memory, a thread 8 queries x
// 8 outputs at a time, two queries per packed FMA.  The sums of the two hidden
// layers run over k in increasing order from the bias, one rounding per term, as
// a scalar evaluation would.  With one query per thread and the weights broadcast, each
// 16-byte shared-memory read fed four FMAs and the reads were the bound (31
// TFLOP/s on a 1080p frame, H = 64); here four of them feed 64.
// The output layer needs no pass of its own over the activations: a thread
// multiplies the 8 x 8 second-layer values that it holds by its outputs'
// columns of W3, and the partial sums of the threads of one query are added
// from shared memory (decode 555 -> 534 us).  An output is its bias plus H / 8
// partial sums, each over eight k from zero: in fp32 like the sums in order, and no
// further from 64 bits (5e-8 relative either way).
// Shared memory: W1^T [16][H], b1, W2^T [H][H], b2, W3 [CP][H], b3[CP], the
// activations [H][kActPitch] (feature columns first; at the end the partial
// sums; the rows' output rows in their pad).  Tiles are split into contiguous
// ranges per CTA so a CTA rarely changes decoder.
constexpr int kActPitch = 132;  // 128 queries and a pad: 16-byte rows, stores of neighbouring rows on other banks

template <int H>
constexpr int fp32_threads() {
  return (kTile / 8) * (H / 8);
}

__device__ __forceinline__ unsigned long long dup2(float x) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %1};" : "=l"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ void fma2(unsigned long long &acc, unsigned long long a, unsigned long long b) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(a), "l"(b));
}
__device__ __forceinline__ unsigned long long pack2(float x, float y) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
  return r;
}
__device__ __forceinline__ float2 unpack2(unsigned long long v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}

// acc[q pair][output] = b[output] + sum_k Wt[k][output] * act[k][query]; this
// thread's queries are q0 .. q0 + 3 and q0 + 64 .. + 67, its outputs o0 .. o0 + 3
// and o0 + H/2 .. + 3, so that a quarter warp's reads are one 128-byte row.
// PAIRS = 2: the first four queries only (the others' sums are zero).
template <int H, int K, int PAIRS>
__device__ __forceinline__ void fp32_layer(const float *Wt, const float *b, const float *act, int q0, int o0,
                                           unsigned long long (&acc)[4][8]) {
#pragma unroll
  for (int o = 0; o < 8; ++o) {
    const unsigned long long v = dup2(b[o0 + (o & 3) + (o >> 2) * (H / 2)]);
#pragma unroll
    for (int p = 0; p < 4; ++p) acc[p][o] = p < PAIRS ? v : 0ull;
  }
#pragma unroll 4
  for (int k = 0; k < K; ++k) {
    const ulonglong2 a0 = *reinterpret_cast<const ulonglong2 *>(act + k * kActPitch + q0);
    ulonglong2 a1 = make_ulonglong2(0, 0);
    if (PAIRS == 4) a1 = *reinterpret_cast<const ulonglong2 *>(act + k * kActPitch + q0 + 64);
    const float4 w0 = *reinterpret_cast<const float4 *>(Wt + k * H + o0);
    const float4 w1 = *reinterpret_cast<const float4 *>(Wt + k * H + o0 + H / 2);
    const float w[8] = {w0.x, w0.y, w0.z, w0.w, w1.x, w1.y, w1.z, w1.w};
#pragma unroll
    for (int o = 0; o < 8; ++o) {
      const unsigned long long ww = dup2(w[o]);
      fma2(acc[0][o], ww, a0.x);
      fma2(acc[1][o], ww, a0.y);
      if (PAIRS == 4) {
        fma2(acc[2][o], ww, a1.x);
        fma2(acc[3][o], ww, a1.y);
      }
    }
  }
}

// ReLU of a layer's outputs into the activations
template <int H>
__device__ __forceinline__ void fp32_store(const unsigned long long (&acc)[4][8], float *act, int q0, int o0) {
#pragma unroll
  for (int o = 0; o < 8; ++o) {
    float *r = act + (o0 + (o & 3) + (o >> 2) * (H / 2)) * kActPitch + q0;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const float2 x = unpack2(acc[2 * h][o]), y = unpack2(acc[2 * h + 1][o]);
      *reinterpret_cast<float4 *>(r + 64 * h) =
          make_float4(fmaxf(x.x, 0.0f), fmaxf(x.y, 0.0f), fmaxf(y.x, 0.0f), fmaxf(y.y, 0.0f));
    }
  }
}

inline __host__ __device__ size_t fp32_img_floats(uint32_t H, uint32_t C) { return (f32_image_floats(H, C) + 3) / 4 * 4; }
inline __host__ __device__ size_t fp32_smem_bytes(uint32_t H, uint32_t C) {
  return (fp32_img_floats(H, C) + (size_t)H * kActPitch) * 4;
}

template <int H, int CP>
__global__ void __launch_bounds__(fp32_threads<H>(), H == 64 ? 4 : 1) k_decode_fp32(Assets A, WeightImages W, Buckets B,
                                                                                   float *out,
                                                                                   unsigned long long *err) {
  extern __shared__ float4 smem4[];
  float *sw = reinterpret_cast<float *>(smem4);
  const float *W1 = sw, *b1 = W1 + H * 16, *W2 = b1 + H, *b2 = W2 + H * H, *W3 = b2 + H, *b3 = W3 + H * CP;
  const uint32_t D = A.num_decoders, C = W.out_dim;
  float *act = sw + fp32_img_floats(H, C);
  // the rows' output rows, in the activations' pad columns: 512 bytes more and
  // only three CTAs of H = 64 fit an SM
  auto row_slot = [&](int i) { return reinterpret_cast<uint32_t *>(act + (i >> 2) * kActPitch + kTile + (i & 3)); };
  constexpr uint32_t kNone = 0xFFFFFFFFu;  // never an output row
  const uint32_t T = __ldg(B.meta);
  const bool copied = rows_copied(B, D);
  const uint32_t t0 = (uint32_t)((unsigned long long)T * blockIdx.x / gridDim.x);
  const uint32_t t1 = (uint32_t)((unsigned long long)T * (blockIdx.x + 1) / gridDim.x);
  const size_t img_floats = f32_image_floats(H, C);
  const int r = threadIdx.x & (kTile - 1);
  const int q0 = ((threadIdx.x / 32 % 2) * 8 + threadIdx.x % 8) * 4, o0 = (threadIdx.x / 64 * 4 + threadIdx.x / 8 % 4) * 4;
  uint32_t cur = 0xFFFFFFFFu;
  for (uint32_t t = t0; t < t1; ++t) {
    uint32_t dec, start, len;
    tile_info(B.meta, D, t, dec, start, len);
    __syncthreads();  // the previous tile has been written
    if (dec != cur && dec < D) {
      const float4 *src = reinterpret_cast<const float4 *>(W.f32 + (size_t)dec * W.f32_stride);
      for (uint32_t i = threadIdx.x; i < img_floats / 4; i += blockDim.x) smem4[i] = __ldg(src + i);
      cur = dec;
    }
    if (threadIdx.x < kTile) {  // one query per thread: its features, or zeros
      const bool valid = (uint32_t)r < len;
      ntc_query q;
      uint32_t oi = 0;
      bool bad = false;
      if (valid) {
        bucket_row(B, copied, start + r, oi, q);
        bad = dec == D || query_bad(A, q);
      }
      count_bad(valid && bad, err);
      float f[kInDim];
#pragma unroll
      for (int k = 0; k < kInDim; ++k) f[k] = 0.0f;
      if (valid && bad)
        for (uint32_t c = 0; c < C; ++c) out[(size_t)oi * C + c] = __int_as_float(0x7fc00000);
      if (valid && !bad) query_features(A, q, f);
#pragma unroll
      for (int k = 0; k < kInDim; ++k) act[k * kActPitch + r] = f[k];
      *row_slot(r) = valid && !bad ? oi : kNone;
    }
    if (dec >= D) continue;  // every row was bad
    // This warp's queries are w0 .. w0 + 31 and w0 + 64 .. + 95; short tiles do
    // without the products past their end.  4,095 decoders with 20,000 queries, a
    // call at H = 64, 9 channels: 234 us with every tile multiplied in full, 172
    // this way (one query per thread: 207); 16 with 300,000: 121 and 118.
    const uint32_t w0 = threadIdx.x / 32 % 2 * 32;
    const bool some = w0 < len, both = w0 + 64 < len;
    auto layer = [&](auto k, const float *Wt, const float *b, unsigned long long (&acc)[4][8]) {
      if (both) fp32_layer<H, decltype(k)::value, 4>(Wt, b, act, q0, o0, acc);
      else if (some) fp32_layer<H, decltype(k)::value, 2>(Wt, b, act, q0, o0, acc);
    };
    __syncthreads();
    unsigned long long acc[4][8];
    layer(std::integral_constant<int, kInDim>(), W1, b1, acc);
    __syncthreads();
    if (some) fp32_store<H>(acc, act, q0, o0);
    __syncthreads();
    layer(std::integral_constant<int, H>(), W2, b2, acc);
#pragma unroll
    for (int o = 0; o < 8; ++o)
#pragma unroll
      for (int p = 0; p < 4; ++p) {
        const float2 x = unpack2(acc[p][o]);
        acc[p][o] = pack2(fmaxf(x.x, 0.0f), fmaxf(x.y, 0.0f));
      }
    const uint32_t oi = *row_slot(r);
    constexpr int kParts = H / 8, kO = 8 * kTile / fp32_threads<H>();  // partial sums of a query; outputs a thread adds up
    const int part = o0 / 4, c0 = (threadIdx.x / kTile) * kO;
#pragma unroll
    for (int cb = 0; cb < CP; cb += 8) {  // eight output channels at a time
      __syncthreads();  // the activations, or the previous channels' sums, have been read
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        if (!some) break;
        const float4 wa = *reinterpret_cast<const float4 *>(W3 + (cb + c) * H + o0);
        const float4 wb = *reinterpret_cast<const float4 *>(W3 + (cb + c) * H + o0 + H / 2);
        const float w[8] = {wa.x, wa.y, wa.z, wa.w, wb.x, wb.y, wb.z, wb.w};
        unsigned long long y[4] = {0, 0, 0, 0};
#pragma unroll
        for (int o = 0; o < 8; ++o) {
          const unsigned long long ww = dup2(w[o]);
#pragma unroll
          for (int p = 0; p < 4; ++p) fma2(y[p], ww, acc[p][o]);
        }
        float *to = act + (part * 8 + c) * kActPitch + q0;
        *reinterpret_cast<ulonglong2 *>(to) = make_ulonglong2(y[0], y[1]);
        *reinterpret_cast<ulonglong2 *>(to + 64) = make_ulonglong2(y[2], y[3]);
      }
      __syncthreads();
      float o[kO];
#pragma unroll
      for (int c = 0; c < kO; ++c) o[c] = b3[cb + c0 + c];
#pragma unroll
      for (int s = 0; s < kParts; ++s)
#pragma unroll
        for (int c = 0; c < kO; ++c) o[c] += act[(s * 8 + c0 + c) * kActPitch + r];
      if (oi != kNone) {
        float *o_row = out + (size_t)oi * C;
#pragma unroll
        for (int c = 0; c < kO; ++c)
          if (cb + c0 + c < (int)C) o_row[cb + c0 + c] = 1.0f / (1.0f + expf(-o[c]));
      }
    }
  }
}

__global__ void k_debug_taps(Assets A, const ntc_query *qs, size_t n, unsigned long long *idx,
                             float *w, float *t_out) {
  const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const ntc_query q = load_query(qs + i);
  const uint32_t L = A.num_levels;
  unsigned long long *I = idx + i * L * 8;
  float *Wt = w + i * L * 8;
  for (uint32_t e = 0; e < L * 8; ++e) {
    I[e] = ~0ull;
    Wt[e] = 0.0f;
  }
  t_out[i] = 0.0f;
  if (query_bad(A, q)) return;
  float t;
  const int lo = select_mip(q.lod, A.num_mips, t);
  t_out[i] = t;
  const GridDesc *g = A.grids + (size_t)q.set_id * L * A.num_mips;
  for (uint32_t k = 0; k < L; ++k) {
    unsigned long long ix[4];
    float wt[4];
    grid_taps(g[k * A.num_mips + lo], q.u, q.v, A.address_mode, ix, wt);
    for (int p = 0; p < 4; ++p) {
      I[k * 8 + p] = ix[p];
      Wt[k * 8 + p] = wt[p];
    }
    if (t > 0.0f) {
      grid_taps(g[k * A.num_mips + lo + 1], q.u, q.v, A.address_mode, ix, wt);
      for (int p = 0; p < 4; ++p) {
        I[k * 8 + 4 + p] = ix[p];
        Wt[k * 8 + 4 + p] = wt[p];
      }
    }
  }
}

// The MLP input of every query: the standard kernels' feature code for the
// standard input (2 levels x 8 channels), the general one otherwise.
__global__ void k_debug_features(Assets A, const ntc_query *qs, size_t n, float *f_out) {
  const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const ntc_query q = load_query(qs + i);
  const uint32_t in = A.num_levels * A.channels + 4 * A.pe_frequencies;
  const bool standard = A.num_levels == kLevels && A.channels == kChannels && A.pe_frequencies == 0;
  float f[kGenMaxIn];
  if (query_bad(A, q)) {
#pragma unroll
    for (int c = 0; c < kGenMaxIn; ++c) f[c] = __int_as_float(0x7fc00000);
  } else if (standard) {
    float s[kInDim];
    query_features(A, q, s);
#pragma unroll
    for (int c = 0; c < kGenMaxIn; ++c) f[c] = c < kInDim ? s[c] : 0.0f;
  } else {
    gen_features(A, A.grids, q, f);
  }
#pragma unroll
  for (int c = 0; c < kGenMaxIn; ++c)
    if (c < (int)in) f_out[i * in + c] = f[c];
}

template <typename T>
__device__ __forceinline__ uint16_t to_bits(float x);
template <>
__device__ __forceinline__ uint16_t to_bits<__half>(float x) {
  return __half_as_ushort(__float2half_rn(x));
}
template <>
__device__ __forceinline__ uint16_t to_bits<__nv_bfloat16>(float x) {
  return __bfloat16_as_ushort(__float2bfloat16_rn(x));
}

// One CTA per decoder: fp32 weights (W1,b1,W2,b2,W3,b3) -> mma image and fp32 image.
template <typename T>
__global__ void k_pack(const float *w32, uint32_t H, uint32_t C, uint8_t *mma, size_t mma_stride,
                       float *f32, size_t f32_stride) {
  const uint32_t d = blockIdx.x;
  const size_t P = (size_t)H * 17 + (size_t)H * (H + 1) + (size_t)C * (H + 1);
  const float *p = w32 + (size_t)d * P;
  const float *W1 = p, *b1 = W1 + H * 16, *W2 = b1 + H, *b2 = W2 + (size_t)H * H, *W3 = b2 + H,
              *b3 = W3 + (size_t)C * H;
  // mma image
  uint16_t *m = reinterpret_cast<uint16_t *>(mma + (size_t)d * mma_stride);
  uint16_t *W1p = m, *W2p = W1p + H * 24, *W3p = W2p + (size_t)H * (H + 8);
  float *bias = reinterpret_cast<float *>(W3p + 16 * (H + 8));
  for (uint32_t i = threadIdx.x; i < H * 24; i += blockDim.x) {
    uint32_t r = i / 24, c = i % 24;
    W1p[i] = c < 16 ? to_bits<T>(W1[r * 16 + c]) : 0;
  }
  for (uint32_t i = threadIdx.x; i < H * (H + 8); i += blockDim.x) {
    uint32_t r = i / (H + 8), c = i % (H + 8);
    W2p[i] = c < H ? to_bits<T>(W2[(size_t)r * H + c]) : 0;
  }
  for (uint32_t i = threadIdx.x; i < 16 * (H + 8); i += blockDim.x) {
    uint32_t r = i / (H + 8), c = i % (H + 8);
    W3p[i] = (r < C && c < H) ? to_bits<T>(W3[(size_t)r * H + c]) : 0;
  }
  for (uint32_t i = threadIdx.x; i < 2 * H + 16; i += blockDim.x)
    bias[i] = i < H ? b1[i] : (i < 2 * H ? b2[i - H] : (i - 2 * H < C ? b3[i - 2 * H] : 0.0f));
  // fp32 image
  const uint32_t CP = out_pad(C);
  float *f = f32 + (size_t)d * f32_stride;
  float *fW1 = f, *fb1 = fW1 + H * 16, *fW2 = fb1 + H, *fb2 = fW2 + (size_t)H * H, *fW3 = fb2 + H,
        *fb3 = fW3 + (size_t)H * CP;
  for (uint32_t i = threadIdx.x; i < H * 16; i += blockDim.x) fW1[i] = W1[(i % H) * 16 + i / H];
  for (uint32_t i = threadIdx.x; i < H; i += blockDim.x) {
    fb1[i] = b1[i];
    fb2[i] = b2[i];
  }
  for (uint32_t i = threadIdx.x; i < H * H; i += blockDim.x) fW2[i] = W2[(size_t)(i % H) * H + i / H];
  for (uint32_t i = threadIdx.x; i < H * CP; i += blockDim.x) fW3[i] = i / H < C ? W3[i] : 0.0f;
  for (uint32_t i = threadIdx.x; i < CP; i += blockDim.x) fb3[i] = i < C ? b3[i] : 0.0f;
}

template <int H, int CP>
cudaError_t launch_fp32_t(const Assets &A, const WeightImages &W, const Buckets &B, size_t n,
                          float *out, unsigned long long *err, int num_sms, cudaStream_t st) {
  const size_t smem = fp32_smem_bytes(H, W.out_dim);
  constexpr int threads = fp32_threads<H>();
  static PerDevice occ_of;
  const int occ = occ_of.value([&]() {
    cudaFuncSetAttribute(k_decode_fp32<H, CP>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
    const int o = resident_ctas(k_decode_fp32<H, CP>, threads, smem);
    return o < 1 ? 1 : o;
  });
  size_t max_tiles = (n + kTile - 1) / kTile + A.num_decoders + 1;
  size_t grid = (size_t)num_sms * occ;
  if (grid > max_tiles) grid = max_tiles;
  k_decode_fp32<H, CP><<<(unsigned)grid, threads, smem, st>>>(A, W, B, out, err);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_decode_fp32(const Assets &A, const WeightImages &W, const Buckets &B, size_t n,
                               float *out, unsigned long long *err, int num_sms, cudaStream_t st,
                               int *launches) {
  *launches += 1;
  const bool c8 = W.out_dim <= 8;
  if (W.hidden == 64)
    return c8 ? launch_fp32_t<64, 8>(A, W, B, n, out, err, num_sms, st)
              : launch_fp32_t<64, 16>(A, W, B, n, out, err, num_sms, st);
  return c8 ? launch_fp32_t<128, 8>(A, W, B, n, out, err, num_sms, st)
            : launch_fp32_t<128, 16>(A, W, B, n, out, err, num_sms, st);
}

cudaError_t launch_debug_taps(const Assets &A, const ntc_query *q, size_t n, unsigned long long *idx,
                              float *w, float *t, cudaStream_t st, int *launches) {
  *launches += 1;
  k_debug_taps<<<(unsigned)((n + 127) / 128), 128, 0, st>>>(A, q, n, idx, w, t);
  return cudaGetLastError();
}

cudaError_t launch_debug_features(const Assets &A, const ntc_query *q, size_t n, float *f,
                                  cudaStream_t st, int *launches) {
  *launches += 1;
  k_debug_features<<<(unsigned)((n + 127) / 128), 128, 0, st>>>(A, q, n, f);
  return cudaGetLastError();
}

cudaError_t launch_pack_weights(const float *w32, uint32_t D, uint32_t H, uint32_t C, bool bf16,
                                uint8_t *mma, size_t mma_stride, float *f32, size_t f32_stride,
                                uint8_t *tc, size_t tc_stride, cudaStream_t st) {
  if (bf16)
    k_pack<__nv_bfloat16><<<D, 256, 0, st>>>(w32, H, C, mma, mma_stride, f32, f32_stride);
  else
    k_pack<__half><<<D, 256, 0, st>>>(w32, H, C, mma, mma_stride, f32, f32_stride);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  return launch_pack_tc(w32, D, H, C, bf16, tc, tc_stride, st);
}

}  // namespace ntc
