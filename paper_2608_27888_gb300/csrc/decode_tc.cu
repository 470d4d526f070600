// tcgen05 / TMEM gather-decode (sm_103a): the production instantiations of
// the kernel in decode_tc.cuh, and the weight-image packing.
#include "decode_tc.cuh"

namespace ntc {

size_t tc_image_bytes(uint32_t H) { return pipe_image_bytes(kInDim, H, 2); }

// One CTA per decoder: fp32 weights -> the shared-memory image of the tcgen05
// kernel (each layer's bias, in kBiasParts parts, at the start of an extra
// 16-wide K block).
template <typename T>
__global__ void k_pack_tc(const float *w32, uint32_t H, uint32_t C, uint8_t *tc, size_t tc_stride) {
  const uint32_t d = blockIdx.x;
  const size_t P = (size_t)H * 17 + (size_t)H * (H + 1) + (size_t)C * (H + 1);
  const float *p = w32 + (size_t)d * P;
  const float *W1 = p, *b1 = W1 + H * 16, *W2 = b1 + H, *b2 = W2 + (size_t)H * H, *W3 = b2 + H,
              *b3 = W3 + (size_t)C * H;
  uint8_t *img = tc + (size_t)d * tc_stride;
  // W [rows][in] and b [rows] (zeros beyond `real` rows) -> [rows][in + 16] at base
  auto layer = [&](uint8_t *base, uint32_t rows, uint32_t real, uint32_t in, const float *W, const float *b) {
    const uint32_t K = in + 16;
    for (uint32_t i = threadIdx.x; i < rows * K; i += blockDim.x) {
      const uint32_t r = i / K, k = i % K;
      T v = T(0.0f);
      if (r < real && k < in) v = T(W[(size_t)r * in + k]);
      else if (r < real && k < in + kBiasParts) v = bias_part<T>(b[r], k - in);
      *reinterpret_cast<T *>(base + core_off(r, k, K)) = v;
    }
  };
  uint8_t *i2 = img + (size_t)H * kTcKA * 2, *i3 = i2 + (size_t)H * (H + 16) * 2;
  layer(img, H, H, 16, W1, b1);
  layer(i2, H, H, H, W2, b2);
  layer(i3, 16, C, H, W3, b3);
}

cudaError_t launch_pack_tc(const float *w32, uint32_t D, uint32_t H, uint32_t C, bool bf16,
                           uint8_t *tc, size_t tc_stride, cudaStream_t st) {
  if (bf16) k_pack_tc<__nv_bfloat16><<<D, 256, 0, st>>>(w32, H, C, tc, tc_stride);
  else k_pack_tc<__half><<<D, 256, 0, st>>>(w32, H, C, tc, tc_stride);
  return cudaGetLastError();
}

cudaError_t launch_decode_tc(const Assets &A, const WeightImages &W, const Buckets &B, size_t n,
                             void *out, unsigned long long *err, unsigned int *status, bool bf16,
                             int num_sms, cudaStream_t st, int *launches) {
  *launches += 1;
  return dispatch_tm<false>(A, W, B, n, out, err, status, bf16, num_sms, st, nullptr);
}

}  // namespace ntc
