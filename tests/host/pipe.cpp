// The tensor-core pipeline's own roles (decode_pipe.cuh, included unchanged) on
// host threads: one thread per warp, the mbarriers, tensor memory, the tensor
// core and the copy engine modelled here.  A tensor-memory column holds the number
// of the tile whose data it would hold, so every MMA, conversion and output row
// can be checked for the tile and the decoder that it works on.
//
// usage: pipe MODE H GENERAL NL GRID CTA SEED BAD TILES_OF_DECODER...
//   MODE run: all roles; silent-dispatcher, silent-loader, silent-producer: that
//   role never starts, so that the others' waits run out.
// usage: pipe bias BITS...: what the bias block of an fp32 bias adds up to, in fp16
//   and in bf16 (hexadecimal bits in, exact decimal sums out)
// Prints one line per violation, and "done".
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#include <atomic>
#include <chrono>
#include <deque>
#include <mutex>
#include <random>
#include <string>
#include <thread>
#include <vector>

#undef __device__
#undef __host__
#undef __forceinline__
#define __device__
#define __host__
#define __forceinline__ inline
struct Dim {
  uint32_t x;
};
static thread_local Dim threadIdx, blockIdx, gridDim, blockDim;

namespace host {
constexpr uint32_t kSmem = 256 * 1024;
alignas(128) static uint8_t smem[kSmem];
static std::atomic<uint32_t> tmem[512];
static std::atomic<int> violations;
static std::mutex lock;
static bool timeouts;  // whether time passes for the bounded waits
static std::atomic<uint64_t> now;
static uint32_t bars_at, img_pitch, images, img_bytes;
static std::atomic<int> image_of[8];  // decoder in an image, -1 while it is loading
static std::vector<uint32_t> decoder;  // of each local tile
static unsigned int status_word;

template <typename... A>
void bad(const char *f, A... a) {
  std::lock_guard<std::mutex> g(lock);
  printf(f, a...);
  printf("\n");
  ++violations;
}

struct Barrier {
  uint32_t count = 0, pending = 0, phase = 0, tx = 0;
};
static Barrier bars[64];
static Barrier *barrier(uint32_t at, const char *what) {
  if (at < bars_at || at >= bars_at + 64 * 8 || (at - bars_at) % 8) {
    bad("%s: no barrier at %u", what, at);
    return nullptr;
  }
  return bars + (at - bars_at) / 8;
}
static void settle(Barrier *b) {
  if (b->pending == 0 && b->tx == 0) b->pending = b->count, ++b->phase;
}
static void arrive(uint32_t at, const char *what) {
  Barrier *b = barrier(at, what);
  if (!b) return;
  std::lock_guard<std::mutex> g(lock);
  if (b->pending == 0) {
    printf("%s: one arrival too many at barrier %d\n", what, (int)(b - bars));
    ++violations;
    return;
  }
  --b->pending;
  settle(b);
}

// The tensor core, one queue per issuer, and the copy engine: threads that take
// their work in order, some time after it was issued.
struct Op {
  int kind;  // 0 MMA, 1 commit, 2 copy
  uint32_t a, b, c, d;
};
static std::deque<Op> queue[3];
static std::mutex qlock;
static std::atomic<bool> stop_engines;
static thread_local int my_queue = 0;
static void push(int q, Op o) {
  std::lock_guard<std::mutex> g(qlock);
  queue[q].push_back(o);
}
static void engine(int q, unsigned seed) {
  std::mt19937 rng(seed + q);
  for (;;) {
    Op o;
    {
      std::lock_guard<std::mutex> g(qlock);
      if (queue[q].empty()) {
        if (stop_engines) return;
        o.kind = -1;
      } else {
        o = queue[q].front();
        queue[q].pop_front();
      }
    }
    for (unsigned i = rng() % 4; i; --i) std::this_thread::yield();
    if (o.kind == 0) {  // d[a] from operand column b and the image at c; d: accumulate
      const uint32_t image = o.c / img_pitch;
      if (image >= images || o.c % img_pitch >= img_bytes) {
        bad("an MMA reads shared memory at %u, outside the images", o.c);
        continue;
      }
      if (o.d) continue;  // a later K step
      const uint32_t tile = tmem[o.b];
      if (timeouts) continue;
      if (tile >= decoder.size()) bad("an MMA reads column %u, which holds no tile", o.b);
      else if (image_of[image] != (int)decoder[tile])
        bad("tile %u of decoder %u is multiplied by image %u, decoder %d", tile, decoder[tile], image, (int)image_of[image]);
      tmem[o.a] = tile;
    } else if (o.kind == 1) {
      arrive(o.a, "commit");
    } else if (o.kind == 2) {  // decoder a into image b, then bytes c of barrier d
      image_of[o.b] = (int)o.a;
      Barrier *x = barrier(o.d, "copy");
      std::lock_guard<std::mutex> g(lock);
      if (x) x->tx -= o.c, settle(x);
    } else {
      std::this_thread::yield();
    }
  }
}
}  // namespace host

#include "decode_pipe.cuh"  // (a copy, beside the host tcgen05.cuh and the parts of ntc_internal.cuh that it uses)

using namespace ntc;

template <int H, int NP, int T, int K1C, int NLC>
static int run(const std::string &mode, uint32_t NL, uint32_t grid, uint32_t cta, unsigned seed, uint32_t bad_tiles,
               const std::vector<uint32_t> &tiles) {
  using P = Pipe<H, false, NP, 2, T, K1C, NLC>;
  const uint32_t D = (uint32_t)tiles.size(), k1 = K1C ? (uint32_t)K1C : 48u;
  std::vector<uint32_t> meta(1 + 2 * (D + 2) + 2), perm;
  uint32_t seg = 0, tst = 0;
  for (uint32_t d = 0; d <= D; ++d) {
    meta[1 + d] = seg, meta[1 + D + 2 + d] = tst;
    const uint32_t t = d < D ? tiles[d] : bad_tiles;
    seg += t ? t * kTile - (d * 37) % kTile : 0, tst += t;  // a ragged last tile
  }
  meta[1 + D + 1] = seg, meta[1 + D + 2 + D + 1] = tst, meta[0] = tst;
  Buckets B{};
  B.meta = meta.data();
  const uint32_t stages = pipe_columns(H, T, k1, NP) <= 512 ? NP : 2;
  uint32_t ns = K1C ? (uint32_t)T : 4;  // the launches' rule
  auto args = [&] { return pipe_args(nullptr, 1, k1, H, NLC ? NLC : NL, ns, NP, stages, 0, D, 9, 0, nullptr, seg); };
  PipeArgs A = args();
  while (!K1C && H == 128 && ns > 1 && A.sm.total > 232448) --ns, A = args();
  memset(host::smem, 0xEE, sizeof host::smem);  // what an earlier kernel left
  host::bars_at = A.sm.bars, host::img_pitch = A.sm.img_pitch, host::images = A.ns, host::img_bytes = A.img_bytes;
  for (auto &i : host::image_of) i = -1;
  blockIdx.x = cta, gridDim.x = grid, blockDim.x = P::kThreads;
  auto constructed = [&](uint32_t thread) {
    threadIdx.x = thread;
    const GridDesc *grids = nullptr;
    return P(A, host::smem, B, D, &host::status_word, grids, 0);
  };
  constructed(0);  // (allocates tensor memory)
  for (uint32_t i = P::kThreads; i-- > 1;) constructed(i);  // every thread's part of the set-up
  const P first = constructed(0);
  {
    TileWalk w;
    for (uint32_t k = 0; k < first.K; ++k) {
      uint32_t d, st, len;
      w.at(first.seg, first.tst, D, first.tile(k), d, st, len);
      if (d >= D != (k >= first.Kg)) host::bad("tile %u: decoder %u, %u good tiles", k, d, first.Kg);
      host::decoder.push_back(d);
    }
  }
  auto warp_of = [&](int warp, auto body) {
    return std::thread([&, warp, body] {
      blockIdx.x = cta, gridDim.x = grid, blockDim.x = P::kThreads, threadIdx.x = (uint32_t)warp * 32;
      P p = first;
      p.warp = warp, p.lane = 0;
      body(p);
    });
  };
  std::vector<std::thread> t, engines;
  for (int q = 0; q < 3; ++q) engines.emplace_back(host::engine, q, seed);
  const std::string silent = mode == "run" ? "" : mode.substr(7);
  for (int w = 0; w < NP * 4 && silent != "producer"; ++w)
    t.push_back(warp_of(w, [&](const P &p) {
      const uint32_t pr = (uint32_t)p.warp / 4;
      for (uint32_t k = pr, j = 0; k < p.Kg && !p.wait.stopped(); k += NP, ++j) {
        uint32_t a[K1C ? K1C / 2 : 24];
        for (auto &x : a) x = k;  // the tile's number for its features
        p.hand_over(pr, j, k, threadIdx.x & 127, a, k);
      }
    }));
  for (int w = 0; w < 8; ++w) t.push_back(warp_of(P::kWarpE + w, [&](const P &p) { p.template convert_tiles<0>((p.warp - P::kWarpE) >> 2); }));
  for (int w = 0; w < 4; ++w)
    t.push_back(warp_of(P::kWarpW + w, [&](const P &p) {  // as the writer hands slots on
      for (uint32_t k = 0; k < p.Kg && !p.wait.stopped(); ++k) {
        const bool there = p.wait(p.ofull_bar(k % T), (k / T) & 1);
        const uint32_t row = p.oidx(k)[threadIdx.x & 127], got = host::tmem[p.t_out(k % T)];
        if (there && !host::timeouts && (row != k || got != k))
          host::bad("tile %u: the writer finds row %u and outputs of tile %u", k, row, got);
        mbar_arrive(p.oempty_bar(k % T));
      }
    }));
  for (int e = 0; e < 2; ++e) t.push_back(warp_of(P::kWarpM + e, [&, e](const P &p) { host::my_queue = e; p.issuer(e); }));
  if (silent != "loader") t.push_back(warp_of(P::kWarpM + 2, [&](const P &p) { p.loader(); }));
  if (silent != "dispatcher") t.push_back(warp_of(P::kWarpM + 3, [&](const P &p) { p.dispatcher(); }));
  for (auto &x : t) x.join();
  host::stop_engines = true;
  for (auto &x : engines) x.join();
  printf("tiles %u images %u stages %u status %u\n", first.Kg, A.ns, first.stages(), host::status_word);
  printf(host::violations ? "%d violations\n" : "done\n", (int)host::violations);
  return 0;
}

template <typename V>
static double block_sum(float b) {
  constexpr bool bf16 = std::is_same<V, __nv_bfloat16>::value;
  double sum = 0;
  for (uint32_t j = 0; j < kBiasParts; ++j) {
    const uint32_t one = bias_ones<bf16>(j & ~1u) >> 16 * (j & 1) & 0xFFFF;
    const float column = bf16 ? (float)__nv_bfloat16(__nv_bfloat16_raw{(unsigned short)one}) : (float)__half(__half_raw{(unsigned short)one});
    sum += (double)column * (double)(float)bias_part<V>(b, j);
  }
  return sum;
}

int main(int argc, char **argv) {
  const std::string mode = argv[1];
  if (mode == "bias") {
    for (int i = 2; i < argc; ++i) {
      const uint32_t bits = (uint32_t)strtoul(argv[i], nullptr, 16);
      float b;
      memcpy(&b, &bits, 4);
      printf("%.17g %.17g\n", block_sum<__half>(b), block_sum<__nv_bfloat16>(b));
    }
    return 0;
  }
  const int H = atoi(argv[2]), general = atoi(argv[3]);
  const uint32_t NL = (uint32_t)atoi(argv[4]), grid = (uint32_t)atoi(argv[5]), cta = (uint32_t)atoi(argv[6]);
  const unsigned seed = (unsigned)atoi(argv[7]);
  const uint32_t bad = (uint32_t)atoi(argv[8]);
  std::vector<uint32_t> tiles;
  for (int i = 9; i < argc; ++i) tiles.push_back((uint32_t)atoi(argv[i]));
  host::timeouts = mode != "run";
  if (!general && H == 64) return run<64, 4, 4, 16, 2>(mode, NL, grid, cta, seed, bad, tiles);
  if (!general) return run<128, 4, 2, 16, 2>(mode, NL, grid, cta, seed, bad, tiles);
  if (general == 8 && H == 64) return run<64, 4, 4, 0, 0>(mode, NL, grid, cta, seed, bad, tiles);
  if (general == 16 && H == 64) return run<64, 2, 4, 0, 0>(mode, NL, grid, cta, seed, bad, tiles);
  if (general == 8) return run<128, 4, 2, 0, 0>(mode, NL, grid, cta, seed, bad, tiles);
  return run<128, 2, 2, 0, 0>(mode, NL, grid, cta, seed, bad, tiles);
}
