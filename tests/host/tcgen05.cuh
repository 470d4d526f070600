// Host versions of tcgen05.cuh's helpers (see pipe.cpp); "warps" of one thread.
#pragma once

#include "../include/ntc.h"

namespace ntc {

template <typename V>
inline V __shfl_sync(unsigned, V v, int) {
  return v;
}
inline bool __all_sync(unsigned, bool x) { return x; }
inline uint32_t ld_word(const uint32_t *p) { return *p; }
inline float __uint_as_float(uint32_t) { return 0.0f; }
inline uint32_t min(uint32_t a, uint32_t b) { return a < b ? a : b; }
constexpr int kTile = NTC_TILE_ROWS;

}  // namespace ntc

#include "parts.cuh"  // GridDesc, Buckets and TileWalk of ntc_internal.cuh

namespace ntc {

inline bool rows_copied(const Buckets &, uint32_t) { return false; }
inline void put_out(void *, size_t, float, bool) {}

constexpr uint64_t kWaitLimitNs = 200ull * 1000ull * 1000ull;

inline uint32_t saddr(const void *p) { return (uint32_t)((const uint8_t *)p - host::smem); }
inline uint64_t global_ns() { return host::timeouts ? host::now += 1000 * 1000 : 0; }
inline bool elect_one() { return true; }
inline uint32_t uniform(uint32_t x) { return x; }
inline void fence_before() {}
inline void fence_after() {}
inline void __syncwarp() {}
inline void __syncthreads() {}
inline void pdl_wait() {}
inline void atomicOr(unsigned int *p, unsigned int v) { *p |= v; }

inline void mbar_init(uint32_t bar, uint32_t count) {
  if (host::Barrier *b = host::barrier(bar, "init")) b->count = b->pending = count;
}
inline void mbar_init_fence() {}
inline bool mbar_try_wait(uint32_t bar, uint32_t parity) {
  std::this_thread::yield();
  host::Barrier *b = host::barrier(bar, "wait");
  std::lock_guard<std::mutex> g(host::lock);
  return !b || (b->phase & 1) != parity;
}
inline bool mbar_wait(uint32_t bar, uint32_t parity) {
  const uint64_t t0 = global_ns();
  while (!mbar_try_wait(bar, parity))
    if (global_ns() - t0 > kWaitLimitNs) return false;
  return true;
}
inline void mbar_arrive(uint32_t bar) { host::arrive(bar, "arrive"); }

inline void bulk_g2s(uint32_t dst, const void *src, uint32_t bytes, uint32_t bar) {
  // src: the images are one byte apart here, so it is the decoder's number
  const uint32_t image = dst / host::img_pitch;
  host::image_of[image] = -1;
  if (host::Barrier *b = host::barrier(bar, "expect")) {
    std::lock_guard<std::mutex> g(host::lock);
    b->tx += bytes, --b->pending;
  }
  host::push(2, {2, (uint32_t)(uintptr_t)src, image, bytes, bar});
}

inline void tmem_alloc(uint32_t to) { memset(host::smem + to, 0, 4); }
inline void tmem_dealloc(uint32_t) {}
inline void tmem_wait_st() {}
inline void tmem_wait_ld() {}
inline uint32_t column(uint32_t taddr) {
  if ((taddr & 0xFFFF) >= 512) host::bad("tensor memory column %u", taddr & 0xFFFF);
  return taddr & 511;
}
template <int N>
inline void tmem_get(uint32_t taddr, uint32_t (&r)[N]) {
  const uint32_t c = column(taddr + N - 1) - (N - 1);
  for (int i = 0; i < N; ++i) r[i] = host::tmem[c + i];
  for (int i = 1; i < N; ++i) r[i] = r[0];
}
template <int N>
inline void tmem_put(uint32_t taddr, const uint32_t (&r)[N]) {
  const uint32_t c = column(taddr + N - 1) - (N - 1);
  for (int i = 0; i < N; ++i) host::tmem[c + i] = r[i];
}
inline void tmem_ld32(uint32_t a, uint32_t (&r)[32]) { tmem_get(a, r); }
inline void tmem_ld16(uint32_t a, uint32_t (&r)[16]) { tmem_get(a, r); }
inline void tmem_st16(uint32_t a, const uint32_t (&r)[16]) { tmem_put(a, r); }
inline void tmem_st8(uint32_t a, const uint32_t (&r)[8]) { tmem_put(a, r); }

inline uint32_t smem_desc_lo(uint32_t addr) { return (addr >> 4) & 0x3FFFu; }
inline uint32_t smem_desc_hi(uint32_t K) { return K; }
template <bool BF16>
constexpr uint32_t instr_desc(uint32_t N) {
  return N;
}
inline void umma_ta(uint32_t d, uint32_t a, uint32_t b_lo, uint32_t b_hi, uint32_t, uint32_t accum) {
  host::push(host::my_queue, {0, column(d), column(a), (b_lo & 0x3FFFu) << 4, accum});
}
inline void umma_commit(uint32_t bar) { host::push(host::my_queue, {1, bar, 0, 0, 0}); }
template <bool BF16>
inline uint32_t pack_relu(uint32_t lo, uint32_t) {
  return lo;  // the tile's number stays
}
template <bool BF16>
inline uint32_t pack(float, float) {
  return 0;
}

}  // namespace ntc
