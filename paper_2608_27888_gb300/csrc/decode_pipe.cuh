// The tensor-core decode pipeline (sm_103a) shared by the standard and the
// general decoder shapes: one persistent 1,024-thread CTA per SM whose warps
// each do one thing, handing tiles (128 queries of one decoder) on through
// mbarriers only.
//
//   Producers (NP warpgroups; thread = row): gather and blend the latents of
//     one tile each and store the feature row into a tensor-memory stage
//     [128 x K1].  Written by each kernel.
//   Issuers (NE warps): one elected lane issues the MMAs of the tiles
//     k = e mod NE: layer 1 from the stage, further layers from the tile
//     slot's hidden operand, the output layer into the slot's own 16 columns.
//   Converters (NE warpgroups): accumulator -> activation -> fp16/bf16 pairs
//     -> the slot's hidden operand.
//   Writers (one warpgroup): output columns -> sigmoid -> out[row].
//   Loader (one warp): copies the weight images the CTA's tiles need, in tile
//     order, into a ring of P.ns images that every tile shares.
//   Dispatcher (one warp): follows the tiles' decoders for the issuers: a
//     tile's stage counts as full only when its weights are there too, and a
//     word per tile says which image it uses and whether it is the last on it.
//     (Left to the issuers, this bookkeeping made one of them need 2,000 cycles
//     a tile, more than any other role.)
//
// T tiles are in flight, one per slot, D = T / NE of them per converter: it
// goes round its D slots layer by layer, so while it converts one tile the
// tensor pipe multiplies the others.
//
// Every layer's bias is one more K step of its MMA: A is a shared block with
// powers of two in its first K columns (bias_scale), and the weight image's extra
// 16-wide K block holds the fp32 bias split into as many fp16/bf16 parts, each
// divided by its column's power: the accumulator gets the bias to fp32 accuracy,
// and the conversions add nothing.
//
// Tiles: CTA b owns the groups b, b + grid, ... of G neighbouring tiles (G = 4
// for long lists), so at any moment the whole GPU works on neighbouring tiles
// -- one decoder and, in bucket order, one set's latents in L2 -- while a CTA's
// consecutive tiles mostly share their weights.
//
// Every wait is bounded (200 ms of %globaltimer, then the status word is set
// and every role leaves at its next tile); tensor memory is released only after
// each issuer's MMAs and the loader's copies have completed.
#pragma once

#include "tcgen05.cuh"

namespace ntc {

constexpr uint32_t kSmemTileTable = 1024;  // staged when D + 2 <= this
constexpr uint32_t kSmemGrids = 1024;      // staged when S * levels * mips <= this
constexpr uint32_t kOidxRing = 16;         // tiles whose output rows are kept (see Pipe)
constexpr uint32_t kNoRow = 0xFFFFFFFFu;   // never an output row: n <= 2^32 - 256
constexpr uint32_t kBiasParts = 4;         // K columns of a bias block that carry the bias

// Shared memory of one launch, as byte offsets: as little as it needs, since
// what is left of the SM's array is the L1 that holds the gathers.
struct PipeSmem {
  uint32_t img_pitch;  // weight images, one after another from 0
  uint32_t oidx, recs, bars, misc, grids, tiles, rows, total;
  static __host__ __device__ __forceinline__ uint32_t row_words(uint32_t C) { return C | 1u; }  // no bank conflicts
  static PipeSmem plan(uint32_t img_bytes, uint32_t ns, uint32_t producers, uint32_t ngrids, uint32_t D, uint32_t C,
                       bool row_buffer) {
    PipeSmem s;
    s.img_pitch = (img_bytes + 127) / 128 * 128;
    s.oidx = ns * s.img_pitch;
    s.recs = s.oidx + kOidxRing * 128 * 4;
    s.bars = s.recs + producers * 128 * (uint32_t)sizeof(ntc_query);
    s.misc = s.bars + 64 * 8;
    s.grids = s.misc + 128;
    s.tiles = s.grids + (ngrids <= kSmemGrids ? ngrids : 0u) * (uint32_t)sizeof(GridDesc);
    s.rows = s.tiles + (D + 2 <= kSmemTileTable ? 2 * (D + 2) : 0u) * 4;
    // a row buffer per writer warp (its reads may run over by two rows of 32)
    s.total = s.rows + (row_buffer ? (4 * 32 * row_words(C) + 64) * 4 : 0u);
    return s;
  }
};

// The decoder and output of one launch.
struct PipeArgs {
  const uint8_t *img;  // [decoders] weight images, img_stride bytes apart
  size_t img_stride;
  uint32_t img_bytes, ns;          // bytes of an image; images in shared memory
  uint32_t stages;                 // tensor-memory stages (Pipe: NP or fewer, both even)
  uint32_t k1, layers;             // K of layer 1 without its bias block; hidden layers
  uint32_t act, slope2;            // 0 ReLU, 1 LeakyReLU, 2 LeakyReLU with 0 <= slope <= 1 (slope2: in both halves)
  float slope;
  uint32_t out_dim, out_half;
  uint32_t vector_rows;            // rows written as one vector store
  uint32_t narrow;                 // every output element's index fits 32 bits
  PipeSmem sm;
};

inline cudaError_t allow_smem(const void *kernel, size_t bytes) {
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

// Bytes of a weight image: W1 [H][k1 + 16], hidden W [H][H + 16], W_out [16][H + 16].
inline __host__ __device__ size_t pipe_image_bytes(uint32_t k1, uint32_t H, uint32_t layers) {
  return ((size_t)H * (k1 + 16) + (size_t)(layers - 1) * H * (H + 16) + (size_t)16 * (H + 16)) * 2;
}

// Tensor-memory columns: T accumulators of H, T hidden operands of H / 2, the
// stages of K1 / 2, the ones block (8), T output accumulators of 16.
constexpr __host__ __device__ uint32_t pipe_columns(uint32_t H, uint32_t T, uint32_t k1, uint32_t stages) {
  return (T * (H + H / 2) + stages * (k1 / 2) + 8 + 15) / 16 * 16 + 16 * T;
}

// What K column j of the shared A block holds, as a power of two.  A bf16 part
// has fp32's range, and three of them its 24 bits (the fourth is 0).  An fp16 part
// has 11 bits between 2^-14 and 2^16, and steps of 2^-24 below: with these powers a
// bias from 2^-15 to 65,519 * 2^15 (2.1e9) splits exactly, a smaller one to within
// 2^-39; a larger one is infinite.  (Parts that all count once leave up to 2^-25,
// and from 65,520 on they are infinite.)
constexpr __host__ __device__ int bias_scale(bool bf16, uint32_t j) {
  return bf16 ? 0 : j == 0 ? 15 : j == 1 ? 4 : j == 2 ? -7 : -14;
}
// The same as a value of the operand type: two K columns, j and j + 1.
template <bool BF16>
constexpr __host__ __device__ uint32_t bias_ones(uint32_t j) {
  return BF16 ? 0x3F80u | 0x3F80u << 16 : (uint32_t)(bias_scale(false, j) + 15) << 10 | (uint32_t)(bias_scale(false, j + 1) + 15) << 26;
}

namespace {

// A bounded wait whose failure ends the launch: sets the status word and the
// CTA's stop flag.
struct Waits {
  volatile uint32_t *stop;
  unsigned int *status;
  __device__ __forceinline__ bool operator()(uint32_t bar, uint32_t parity) const {
    if (mbar_try_wait(bar, parity)) return true;
    const uint64_t t0 = global_ns();
    while (!mbar_try_wait(bar, parity)) {
      if (*stop) return false;
      if (global_ns() - t0 > kWaitLimitNs) {
        atomicOr(status, 1u);
        *stop = 1;
        return false;
      }
    }
    return true;
  }
  __device__ __forceinline__ bool stopped() const { return uniform(*stop) != 0; }
};

// An output element under a predicate: no branch, so that neighbouring elements
// overlap.
__device__ __forceinline__ void put_elem_if(bool on, float *p, float y) {
  asm volatile("{\n.reg .pred p;\nsetp.ne.u32 p, %2, 0;\n@p st.global.f32 [%0], %1;\n}\n" ::"l"(p), "f"(y),
               "r"((uint32_t)on)
               : "memory");
}
__device__ __forceinline__ void put_elem_if(bool on, __half *p, float y) {
  asm volatile("{\n.reg .pred p;\nsetp.ne.u32 p, %2, 0;\n@p st.global.u16 [%0], %1;\n}\n" ::"l"(p),
               "h"(__half_as_ushort(__float2half_rn(y))), "r"((uint32_t)on)
               : "memory");
}

// A warp's 32 output rows of C elements, from its row buffer (row r of the
// warp at r * PipeSmem::row_words(C)) to out: element k = lane + 32 i of the
// 32 x C block in store i, so that a store covers consecutive elements of a few
// rows.  Stored straight from the accumulator instead, one channel per
// instruction, a nine-channel row's sectors are touched once per channel, 1.5 GB
// through the SM-to-L2 crossbar for a 2160p frame instead of 0.3; but each
// shared-memory or shuffle step of this way queues behind the producers'
// gathers.  At H = 128 the crossbar is what matters (four trilinear 2160p
// frames, nine channels: decode 1,421 -> 1,327 us with the buffer), at H = 64 the
// writers' time per tile (a 2160p frame 350 us with it, 218 without; Sec. 4's
// decoder on 1080p 143 and 86).  Sec. 4's decoder at H = 128, whose gathers are
// half as wide, would be better off without it too (128 x 5 on 1283 x 717: 106 us
// with it, 95 without).
struct RowWriter {
  uint32_t at[16];  // element i: its row in the low 5 bits, its channel from bit 8
  __device__ __forceinline__ RowWriter(uint32_t C, int lane) {
#pragma unroll
    for (uint32_t i = 0; i < 16; ++i) {
      const uint32_t k = (uint32_t)lane + 32 * i, r = k / C;
      at[i] = (r & 31u) | (k - r * C) << 8;
    }
  }
  // narrow: every element's index fits 32 bits
  template <typename E>
  __device__ __forceinline__ void operator()(E *out, const float *rowbuf, uint32_t C, uint32_t oi, bool good, int lane,
                                             bool narrow) const {
    const uint32_t oi0 = __shfl_sync(0xFFFFFFFFu, oi, 0);
    if ((C & 1) && __all_sync(0xFFFFFFFFu, good && oi == oi0 + (uint32_t)lane)) {
      // the rows are side by side: 32 C consecutive elements on both sides
      E *p = out + (size_t)oi0 * C + lane;
#pragma unroll
      for (uint32_t g = 0; g < 16; g += 3) {
        if (g >= C) break;
        float v[3];
#pragma unroll
        for (uint32_t j = 0; j < 3; ++j) v[j] = rowbuf[lane + 32 * (g + j)];
#pragma unroll
        for (uint32_t j = 0; j < 3; ++j) put_elem_if(g + j < C, p + 32 * (g + j), v[j]);
      }
      return;
    }
    const uint32_t even = 1u - (C & 1u);
    const uint32_t base = good ? (narrow ? oi * C : oi) : kNoRow;  // the row's first element, or the row
#pragma unroll
    for (uint32_t g = 0; g < 16; g += 3) {
      if (g >= C) break;
      float v[3];
      uint32_t to[3];
#pragma unroll
      for (uint32_t j = 0; j < 3; ++j) {
        const uint32_t i = g + j < 16 ? g + j : 15, w = at[i];
        to[j] = __shfl_sync(0xFFFFFFFFu, base, w);
        v[j] = rowbuf[(uint32_t)lane + 32 * i + even * (w & 31u)];
      }
#pragma unroll
      for (uint32_t j = 0; j < 3; ++j) {
        const uint32_t i = g + j < 16 ? g + j : 15, ch = at[i] >> 8;
        put_elem_if(g + j < C && to[j] != kNoRow, out + (narrow ? (size_t)(to[j] + ch) : (size_t)to[j] * C + ch), v[j]);
      }
    }
  }
};

// An activated fp16/bf16 pair of accumulator values.  act 2 evaluates
// max(h, slope * h) on the packed pair.
template <bool BF16, int ACT>
__device__ __forceinline__ uint32_t pack_act(uint32_t lo, uint32_t hi, float slope, uint32_t slope2) {
  if (ACT == 0) return pack_relu<BF16>(lo, hi);
  if (ACT == 2) {
    const uint32_t h = pack<BF16>(__uint_as_float(lo), __uint_as_float(hi));
    uint32_t r;
    if (BF16)
      asm("{\n.reg .b32 t;\nmul.rn.bf16x2 t, %1, %2;\nmax.bf16x2 %0, %1, t;\n}" : "=r"(r) : "r"(h), "r"(slope2));
    else
      asm("{\n.reg .b32 t;\nmul.rn.f16x2 t, %1, %2;\nmax.f16x2 %0, %1, t;\n}" : "=r"(r) : "r"(h), "r"(slope2));
    return r;
  }
  const float a = __uint_as_float(lo), b = __uint_as_float(hi);
  return pack<BF16>(a > 0.0f ? a : slope * a, b > 0.0f ? b : slope * b);
}

// The pipeline of one CTA.  K1C, NLC: K of layer 1 and the hidden layers when
// the kernel is compiled for them (0: P.k1, P.layers).
// Handing over: tile k is gathered by producer k mod NP into stage
// k mod stages; full[k mod NP] counts its four warps and the dispatcher, and
// layer 1 of tile k commits to empty[] of the producer of tile k + stages, the
// stage's next.  Issuer e has the tiles k = e mod NE.  Every barrier must have
// waiters that see each of its phases in turn (a parity wait for a phase
// beyond the next returns at once), so NP and the stages are multiples of NE:
// a full[] barrier then belongs to one issuer.  And layer 1 of tile
// k - stages, which lets the producer's warps go on to tile k, comes after
// that of tile k - NP from the same issuer, so no warp arrives for tile k while
// others still have to arrive for tile k - NP.
// Output rows: the producer of tile k writes oidx[k mod 16] once layer 1 of
// tile k - stages has completed, so the output layer of tile k - stages - T was
// issued, so the writers had read tile k - stages - 2T and every tile before
// it: the ring holds stages + 2T <= 12 tiles.
// Weight ring: epoch = the number of decoder changes along the CTA's tiles.  The
// loader reuses an image once its epoch's tiles are done: each issuer's last
// tile on it commits to the image's barrier after its output layer (an issuer
// that has none leaves it to the other one).  The T tiles in flight span at
// most T epochs, so P.ns >= T images never deadlock; with D = 1 an issuer
// holds no tile while it waits for the next one's weights, and any P.ns does.
template <int H, bool BF16, int NP, int NE, int T, int K1C, int NLC>
struct Pipe {
  static constexpr int D = T / NE;
  static_assert(T % NE == 0 && NP % NE == 0 && NE <= 2, "each slot and each full barrier belongs to one issuer");
  static constexpr int kThreads = (NP + NE + 2) * 128;
  static constexpr int kWarpE = NP * 4, kWarpW = kWarpE + NE * 4, kWarpM = kWarpW + 4;  // first warps of the roles
  static_assert(NP <= 8 && NP + 2 * T <= (int)kOidxRing, "output-row ring too short");
  const PipeArgs &P;
  uint8_t *smem;
  uint32_t sbase, tmem;
  Waits wait;
  uint32_t K, Kg;        // local tiles; those before the bad bucket
  uint32_t grid, gshift; // tiles per group = 1 << gshift
  uint32_t gstep, gfirst;
  uint32_t D_;           // decoders
  const uint32_t *seg, *tst;
  uint32_t ident_n;
  int warp, lane;

  __device__ __forceinline__ uint32_t k1() const { return K1C ? (uint32_t)K1C : P.k1; }
  __device__ __forceinline__ uint32_t nl() const { return NLC ? (uint32_t)NLC : P.layers; }
  __device__ __forceinline__ uint32_t stages() const { return K1C ? (uint32_t)NP : P.stages; }
  // barriers
  __device__ __forceinline__ uint32_t bar(uint32_t i) const { return sbase + P.sm.bars + 8 * i; }
  __device__ __forceinline__ uint32_t full_bar(uint32_t p) const { return bar(p); }          // producer p's tile is in its stage
  __device__ __forceinline__ uint32_t empty_bar(uint32_t p) const { return bar(8 + p); }     // producer p's next stage is free
  __device__ __forceinline__ uint32_t acc_bar(uint32_t s) const { return bar(16 + s); }      // a hidden layer's result
  __device__ __forceinline__ uint32_t hid_bar(uint32_t s) const { return bar(20 + s); }      // ... converted
  __device__ __forceinline__ uint32_t ofull_bar(uint32_t s) const { return bar(24 + s); }    // the output layer's result
  __device__ __forceinline__ uint32_t oempty_bar(uint32_t s) const { return bar(28 + s); }   // ... read
  __device__ __forceinline__ uint32_t wfull_bar(uint32_t i) const { return bar(32 + i); }    // a weight image is loaded
  __device__ __forceinline__ uint32_t wempty_bar(uint32_t i) const { return bar(40 + i); }   // ... and free again
  __device__ __forceinline__ uint32_t final_bar(uint32_t e) const { return bar(48 + e); }
  // tensor memory
  __device__ __forceinline__ uint32_t t_acc(uint32_t s) const { return tmem + s * H; }
  __device__ __forceinline__ uint32_t t_hid(uint32_t s) const { return tmem + T * H + s * (H / 2); }
  __device__ __forceinline__ uint32_t t_stage(uint32_t st) const { return tmem + T * (H + H / 2) + st * (k1() / 2); }
  __device__ __forceinline__ uint32_t t_ones() const { return t_stage(stages()); }
  __device__ __forceinline__ uint32_t t_out(uint32_t s) const {
    return tmem + (T * (H + H / 2) + stages() * (k1() / 2) + 8 + 15) / 16 * 16 + 16 * s;
  }
  __device__ __forceinline__ uint32_t lanes() const { return (uint32_t)((warp & 3) * 32) << 16; }
  __device__ __forceinline__ uint32_t *oidx(uint32_t k) const {
    return reinterpret_cast<uint32_t *>(smem + P.sm.oidx) + (k % kOidxRing) * 128;
  }
  // what the dispatcher says of tile k: its image, and (from bit 8) how many
  // commits to the image's barrier follow the tile's output layer
  __device__ __forceinline__ volatile uint32_t *info(uint32_t k) const {
    return reinterpret_cast<volatile uint32_t *>(smem + P.sm.misc) + 4 + k % kOidxRing;
  }
  // global tile of local tile k
  __device__ __forceinline__ uint32_t tile(uint32_t k) const {
    return k + (k >> gshift) * gstep + gfirst;  // ((k >> gshift) * grid + CTA) << gshift, + k mod the group
  }
  // local tiles of a list of n global tiles
  __device__ __forceinline__ uint32_t local(uint32_t n) const {
    const uint32_t groups = (n + (1u << gshift) - 1u) >> gshift;
    if (blockIdx.x >= groups) return 0;
    const uint32_t mine = (groups - blockIdx.x + grid - 1) / grid, last = blockIdx.x + (mine - 1) * grid;
    return (mine << gshift) - (last == groups - 1 ? (groups << gshift) - n : 0u);
  }

  // Everything before the roles part.  grids: the grid table of the latents,
  // returned as its shared-memory copy when that fits.
  __device__ __forceinline__ Pipe(const PipeArgs &args, uint8_t *sm, const Buckets &B, uint32_t decoders,
                                  unsigned int *status, const GridDesc *&grids, uint32_t ngrids)
      : P(args), smem(sm), sbase(saddr(sm)), D_(decoders), ident_n(B.identity_n) {
    warp = (int)uniform(threadIdx.x >> 5);
    lane = threadIdx.x & 31;
    grid = gridDim.x;
    uint32_t *misc = reinterpret_cast<uint32_t *>(smem + P.sm.misc);
    wait.stop = misc + 1;
    wait.status = status;
    for (uint32_t i = threadIdx.x; i < kOidxRing * 128; i += blockDim.x)
      reinterpret_cast<uint32_t *>(smem + P.sm.oidx)[i] = kNoRow;
    // an issuer whose wait for the dispatcher has run out reads its word all the
    // same: until one is written it names image 0 and no commits, so that what it
    // then issues stays inside the images and the barriers
    for (uint32_t i = threadIdx.x; i < kOidxRing; i += blockDim.x) *info(i) = 0;
    if (ngrids <= kSmemGrids) {
      GridDesc *g = reinterpret_cast<GridDesc *>(smem + P.sm.grids);
      for (uint32_t i = blockDim.x - 1 - threadIdx.x; i < ngrids; i += blockDim.x) g[i] = grids[i];
      grids = g;
    }
    // What a call of a few tiles per CTA takes is mostly this set-up, so its parts
    // run side by side: the barriers by a thread of the second and one of the
    // third warp, the allocation by the first, the grid table above by the last
    // (all by the first warp, one after the other, and the divisions below for
    // both lists also where they are the same: a 65,536-query raster 6.2 us of GPU
    // time, this way 5.6).
    if (threadIdx.x == 32) {
      for (uint32_t i = 0; i < 8; ++i) {
        mbar_init(full_bar(i), 5);   // one arrival per producer warp, and the dispatcher's
        mbar_init(empty_bar(i), 1);  // layer 1's commit
        mbar_init(wfull_bar(i), 1);
        mbar_init(wempty_bar(i), NE);  // each issuer's commit
      }
      mbar_init_fence();
    }
    if (threadIdx.x == 64) {
      for (uint32_t i = 0; i < 4; ++i) {
        mbar_init(acc_bar(i), 1);
        mbar_init(hid_bar(i), 4);  // one arrival per converter warp
        mbar_init(ofull_bar(i), 1);
        mbar_init(oempty_bar(i), 4);  // one arrival per writer warp
        mbar_init(final_bar(i), 1);
      }
      misc[1] = 0;
      mbar_init_fence();
    }
    if (warp == 0) tmem_alloc(saddr(misc));
    fence_before();
    __syncthreads();
    fence_after();
    tmem = uniform(*reinterpret_cast<volatile uint32_t *>(misc));
    if (warp < 4) {  // the bias operand
      const uint32_t z[8] = {bias_ones<BF16>(0), bias_ones<BF16>(2), 0u, 0u, 0u, 0u, 0u, 0u};
      tmem_st8(t_ones() + lanes(), z);
      tmem_wait_st();
    }
    // everything above is independent of the bucketing; the tile table is not
    pdl_wait();
    seg = B.meta + 1;
    tst = seg + (D_ + 2);
    if (!ident_n && D_ + 2 <= kSmemTileTable) {
      uint32_t *s_seg = reinterpret_cast<uint32_t *>(smem + P.sm.tiles), *s_tst = s_seg + (D_ + 2);
      for (uint32_t i = threadIdx.x; i < D_ + 2; i += blockDim.x) {
        s_seg[i] = ld_word(seg + i);
        s_tst[i] = ld_word(tst + i);
      }
      seg = s_seg;
      tst = s_tst;
    }
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t all = ident_n ? (ident_n + kTile - 1) / kTile : tst[D_ + 1];
    const uint32_t good = ident_n ? all : tst[D_];  // the bad bucket's tiles come last
    // longer groups share weights better, but leave the last wave emptier.  At
    // H = 128 single tiles are better on long lists where a decoder has four or
    // more per CTA anyway (four trilinear 2160p frames, 8 decoders: 1,511 ->
    // 1,500 us a call; 586 decoders on 1080p: decode 127 us, with groups 88)
    gshift = all >= 64 * grid ? (H == 128 && all / D_ >= 4 * grid ? 0u : 2u) : all >= 24 * grid ? 1u : 0u;
    gstep = (grid - 1) << gshift;
    gfirst = blockIdx.x << gshift;
    if (good == all) {
      K = Kg = local(all);
    } else {
      K = local(all);
      Kg = local(good);
    }
  }

  // The rows of one producer thread, tile by tile (k = p, p + NP, ...): while
  // tile k is gathered, the record of its next tile is on its way to the
  // thread's slot in shared memory (cp.async: no registers) and the output row
  // (perm) of the one after it to a register, so that neither a record nor the
  // perm entry that leads to it is waited for.  Loaded one tile ahead together,
  // they cost a 1080p frame's producers about a quarter of their time.
  struct Rows {
    const Buckets &B;
    TileWalk walk;
    bool copied;
    uint32_t slot;       // shared memory of this thread's record
    uint32_t oi;         // output row of the current tile, or kNoRow past its end
    uint32_t noi, npos;  // of the next tile, and its place in bucket order
    // a row of the bad bucket (set id out of range) needs no flag of its own:
    // query_bad() rejects it
    __device__ __forceinline__ void row_of(const Pipe &q, uint32_t k, uint32_t &oi_, uint32_t &pos) {
      oi_ = kNoRow;
      if (k >= q.K) return;
      uint32_t d, st, len;
      const uint32_t row = threadIdx.x & 127;
      walk.at(q.seg, q.tst, q.D_, q.tile(k), d, st, len);
      if (row >= len) return;
      pos = st + row;
      oi_ = q.ident_n ? pos : ld_word(B.perm + pos);
    }
    __device__ __forceinline__ void request() {  // the next tile's record
      if (noi != kNoRow)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(slot),
                     "l"(copied ? B.sorted + npos : B.queries + noi)
                     : "memory");
    }
    __device__ __forceinline__ Rows(const Pipe &q, const Buckets &b, uint32_t p) : B(b) {
      walk.ident_n = q.ident_n;
      copied = rows_copied(B, q.D_);
      slot = q.sbase + q.P.sm.recs + (p * 128 + (threadIdx.x & 127)) * (uint32_t)sizeof(ntc_query);
      row_of(q, p, noi, npos);
      request();
      oi = noi;
      row_of(q, p + NP, noi, npos);
    }
    // the current tile's record (undefined past the tile's end)
    __device__ __forceinline__ ntc_query record() const {
      asm volatile("cp.async.wait_all;\n" ::: "memory");
      ntc_query r;
      asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];\n"
                   : "=r"(r.set_id), "=f"(r.u), "=f"(r.v), "=f"(r.lod)
                   : "r"(slot)
                   : "memory");
      return r;
    }
    // after record() of tile k has been looked at
    __device__ __forceinline__ void look_ahead(const Pipe &q, uint32_t k, uint32_t &next) {
      request();
      next = noi;
      row_of(q, k + 2 * NP, noi, npos);
    }
  };

  // Ends the CTA: every role has left.
  __device__ __forceinline__ void end() const {
    fence_before();
    __syncthreads();
    if (warp == 0) {
      fence_after();
      tmem_dealloc(tmem);
    }
  }

  // A producer warp has its rows of local tile k (the j-th of its warpgroup
  // p): wait for the stage, store K1 / 2 words a row, hand over.
  template <int NW>
  __device__ __forceinline__ void hand_over(uint32_t p, uint32_t j, uint32_t k, uint32_t row, const uint32_t (&a)[NW],
                                            uint32_t oi) const {
    // the stage's previous tile has left layer 1 (the first `stages` tiles have none)
    const uint32_t n = stages(), st = K1C ? p : k % n;
    wait(empty_bar(p), (p < n ? j + 1 : j) & 1);
    fence_after();
#pragma unroll
    for (int kc = 0; kc < NW / 8; ++kc) {
      if (!K1C && (uint32_t)kc * 16 >= k1()) break;
      uint32_t w[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) w[i] = a[8 * kc + i];
      tmem_st8(t_stage(st) + lanes() + 8 * kc, w);
    }
    tmem_wait_st();
    oidx(k)[row] = oi;
    fence_before();
    __syncwarp();
    if (lane == 0) mbar_arrive(full_bar(p));
  }

  // The decoder of each of the CTA's tiles in turn.
  __device__ __forceinline__ uint32_t decoder_of(TileWalk &walk, uint32_t k) const {
    uint32_t d, st, len;
    walk.at(seg, tst, D_, tile(k), d, st, len);
    return d;
  }

  __device__ __forceinline__ void loader() const {
    TileWalk walk;
    walk.ident_n = ident_n;
    uint32_t e = 0, i = 0, use = 0, dec = 0xFFFFFFFFu;  // images loaded; the ring's next image and its use
    for (uint32_t k = 0; k < Kg; ++k) {
      const uint32_t d = decoder_of(walk, k);
      if (d == dec) continue;
      dec = d;
      if (!uniform(wait(wempty_bar(i), (use & 1) ^ 1))) break;
      if (elect_one()) bulk_g2s(sbase + i * P.sm.img_pitch, P.img + (size_t)d * P.img_stride, P.img_bytes, wfull_bar(i));
      ++e;
      if (++i == P.ns) i = 0, ++use;
    }
    // no copy is in flight when the CTA ends
    for (uint32_t j = e > P.ns ? e - P.ns : 0; j < e; ++j) mbar_wait(wfull_bar(j % P.ns), (j / P.ns) & 1);
  }

  __device__ __forceinline__ void dispatcher() const {
    constexpr uint32_t kNone = 0xFFFFFFFEu;  // never a decoder
    TileWalk walk;
    walk.ident_n = ident_n;
    uint32_t i = 0, use = 0;  // this tile's image and its use
    uint32_t before = kNone, d0 = Kg > 0 ? decoder_of(walk, 0) : kNone, d1 = Kg > 1 ? decoder_of(walk, 1) : kNone;
    for (uint32_t k = 0; k < Kg && !wait.stopped(); ++k) {
      const uint32_t d2 = k + 2 < Kg ? decoder_of(walk, k + 2) : kNone;
      if (k && d0 != before && ++i == P.ns) i = 0, ++use;
      // the last tile on an image commits; with two issuers the last of each
      // does, and an only tile commits for both
      const bool last = d1 != d0;
      uint32_t commits = last;
      if (NE == 2) commits += last ? d0 != before : d2 != d1;
      wait(wfull_bar(i), use & 1);
      const uint32_t p = k % NP, j = k / NP;
      if (j) wait(full_bar(p), (j - 1) & 1);  // this arrival is for the next phase
      if (lane == 0) {
        *info(k) = i | commits << 8;
        mbar_arrive(full_bar(p));
      }
      before = d0, d0 = d1, d1 = d2;
    }
  }

  // Low word of the descriptor of layer l's weights (0: layer 1) of the image
  // the dispatcher named.
  __device__ __forceinline__ uint32_t w_desc(uint32_t word, uint32_t l) const {
    const uint32_t K1 = k1();
    return smem_desc_lo(sbase + (word & 0xFFu) * P.sm.img_pitch +
                        (l ? H * (K1 + 16) + (l - 1) * H * (H + 16) : 0u) * 2);
  }

  __device__ __forceinline__ void issuer(uint32_t e) const {
    const uint32_t own = Kg > e ? (Kg - e + NE - 1) / NE : 0;  // this issuer's tiles
    const uint32_t NL = nl(), K1 = k1();
    constexpr uint32_t id_h = instr_desc<BF16>(H), id_o = instr_desc<BF16>(16);
    const uint32_t hi1 = smem_desc_hi(K1 + 16), hi2 = smem_desc_hi(H + 16);
    const bool leader = elect_one();
    uint32_t said[D];  // per slot of this issuer, what the dispatcher said of its tile
    uint32_t st = e % stages();  // the next layer 1's stage
    auto layer1 = [&](uint32_t k, uint32_t s, uint32_t &word) {  // tile k, into slot s
      wait(full_bar(k % NP), (k / NP) & 1);
      word = uniform(*info(k));
      fence_after();
      const uint32_t d = w_desc(word, 0);
      if (leader) {
        for (uint32_t kq = 0; kq < K1 / 16; ++kq) umma_ta(t_acc(s), t_stage(st) + 8 * kq, d + 16 * kq, hi1, id_h, kq);
        umma_ta(t_acc(s), t_ones(), d + K1, hi1, id_h, 1);  // + bias
        umma_commit(acc_bar(s));
        umma_commit(empty_bar((k + stages()) % NP));
      }
      __syncwarp();
      st += NE;
      if (st >= stages()) st -= stages();
    };
#pragma unroll
    for (uint32_t s_ = 0; s_ < (uint32_t)D; ++s_)
      if (s_ < own) layer1(e + NE * s_, e + NE * s_, said[s_]);
    uint32_t j = 0;  // the slots' uses
    for (uint32_t g = 0; g < own && !wait.stopped(); g += D, ++j) {
      for (uint32_t l = 0; l < NL; ++l) {
        const uint32_t parity = (j * NL + l) & 1;
#pragma unroll
        for (uint32_t s_ = 0; s_ < (uint32_t)D; ++s_) {
          if (g + s_ >= own) break;
          const uint32_t s = e + NE * s_, k = e + NE * (g + s_);
          wait(hid_bar(s), parity);
          fence_after();
          const uint32_t word = said[s_], d = w_desc(word, l + 1);
          if (l + 1 < NL) {
            if (leader) {
#pragma unroll
              for (uint32_t kq = 0; kq < H / 16; ++kq) umma_ta(t_acc(s), t_hid(s) + 8 * kq, d + 16 * kq, hi2, id_h, kq);
              umma_ta(t_acc(s), t_ones(), d + H, hi2, id_h, 1);
              umma_commit(acc_bar(s));
            }
            __syncwarp();
          } else {
            wait(oempty_bar(s), (j & 1) ^ 1);  // the slot's previous outputs have been read
            fence_after();
            if (leader) {
#pragma unroll
              for (uint32_t kq = 0; kq < H / 16; ++kq) umma_ta(t_out(s), t_hid(s) + 8 * kq, d + 16 * kq, hi2, id_o, kq);
              umma_ta(t_out(s), t_ones(), d + H, hi2, id_o, 1);
              umma_commit(ofull_bar(s));
              for (uint32_t c = word >> 8; c; --c) umma_commit(wempty_bar(word & 0xFFu));
            }
            __syncwarp();
            // the slot's next tile; its commit also covers the output layer,
            // which reads the hidden operand that the conversion overwrites
            if (g + s_ + D < own) layer1(k + T, s, said[s_]);
          }
        }
      }
    }
    // no MMA of this warp is in flight when tensor memory is released
    if (leader) umma_commit(final_bar(e));
    __syncwarp();
    mbar_wait(final_bar(e), 0);
  }

  // TMEM accumulator -> activation -> fp16/bf16 pairs -> hidden operand
  template <int ACT>
  __device__ __forceinline__ void convert(uint32_t ta, uint32_t th) const {
    if constexpr (H == 16) {
      uint32_t v[16], p[8];
      tmem_ld16(ta, v);
      tmem_wait_ld();
#pragma unroll
      for (int i = 0; i < 8; ++i) p[i] = pack_act<BF16, ACT>(v[2 * i], v[2 * i + 1], P.slope, P.slope2);
      tmem_st8(th, p);
    } else {
#pragma unroll
      for (int c = 0; c < H; c += 32) {
        uint32_t v[32], p[16];
        tmem_ld32(ta + c, v);
        tmem_wait_ld();
#pragma unroll
        for (int i = 0; i < 16; ++i) p[i] = pack_act<BF16, ACT>(v[2 * i], v[2 * i + 1], P.slope, P.slope2);
        tmem_st16(th + c / 2, p);
      }
    }
    tmem_wait_st();
  }

  __device__ __forceinline__ void converter(uint32_t e) const {  // (a test per value costs as much as the conversion)
    if (K1C || P.act == 0) convert_tiles<0>(e);  // the standard shape has ReLU
    else if (P.act == 2) convert_tiles<2>(e);
    else convert_tiles<1>(e);
  }
  template <int ACT>
  __device__ __forceinline__ void convert_tiles(uint32_t e) const {
    const uint32_t own = Kg > e ? (Kg - e + NE - 1) / NE : 0, NL = nl();
    uint32_t j = 0;  // the slots' uses
    for (uint32_t g = 0; g < own && !wait.stopped(); g += D, ++j) {
      const uint32_t slots = own - g < (uint32_t)D ? own - g : (uint32_t)D;
      for (uint32_t l = 0; l < NL; ++l) {
        const uint32_t parity = (j * NL + l) & 1;
#pragma unroll 1
        for (uint32_t s_ = 0; s_ < slots; ++s_) {
          const uint32_t s = e + NE * s_;
          wait(acc_bar(s), parity);
          fence_after();
          convert<ACT>(t_acc(s) + lanes(), t_hid(s) + lanes());
          fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(hid_bar(s));
        }
      }
    }
  }
  __device__ __forceinline__ void writer(void *out) const {
    const uint32_t row = threadIdx.x & 127, C = P.out_dim;
    float *rowbuf = reinterpret_cast<float *>(smem + P.sm.rows) + (warp & 3) * 32 * PipeSmem::row_words(C);
    const RowWriter write(kRowBuffer ? C : 16u, lane);
    auto sigmoid = [](uint32_t x) {  // 0.5 + 0.5 * tanh(x / 2)
      float th;
      asm("tanh.approx.f32 %0, %1;" : "=f"(th) : "f"(0.5f * __uint_as_float(x)));
      return fmaf(0.5f, th, 0.5f);
    };
    for (uint32_t k = 0; k < Kg && !wait.stopped(); ++k) {
      const uint32_t s = k % T;
      wait(ofull_bar(s), (k / T) & 1);
      fence_after();
      const uint32_t oi = oidx(k)[row];
      uint32_t o[16];
      tmem_ld16(t_out(s) + lanes(), o);
      tmem_wait_ld();
      fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(oempty_bar(s));
      const bool good = oi != kNoRow;
      if (P.vector_rows) {
        float y[8];
#pragma unroll
        for (int c = 0; c < 8; ++c) y[c] = sigmoid(o[c]);
        if (!good) {
        } else if (P.out_half) {  // one 16-byte store per row
          uint32_t h[4];
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const __half2 p = __floats2half2_rn(y[2 * i], y[2 * i + 1]);
            h[i] = *reinterpret_cast<const uint32_t *>(&p);
          }
          asm volatile("st.global.v4.b32 [%0], {%1, %2, %3, %4};\n" ::"l"(reinterpret_cast<__half *>(out) +
                                                                        (size_t)oi * 8),
                       "r"(h[0]), "r"(h[1]), "r"(h[2]), "r"(h[3])
                       : "memory");
        } else {  // one 32-byte store per row
          asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};\n" ::"l"(
                           reinterpret_cast<float *>(out) + (size_t)oi * 8),
                       "f"(y[0]), "f"(y[1]), "f"(y[2]), "f"(y[3]), "f"(y[4]), "f"(y[5]), "f"(y[6]), "f"(y[7])
                       : "memory");
        }
        continue;
      }
      if (!kRowBuffer) {
        if (good)
#pragma unroll
          for (int c = 0; c < 16; ++c)
            if (c < (int)C) put_out(out, (size_t)oi * C + c, sigmoid(o[c]), P.out_half);
        continue;
      }
      const uint32_t row_at = saddr(rowbuf) + lane * PipeSmem::row_words(C) * 4;
#pragma unroll
      for (int h = 0; h < 16; h += 8) {
        if (h >= (int)C) break;
        float y[8];
#pragma unroll
        for (int c = 0; c < 8; ++c) y[c] = sigmoid(o[h + c]);
#pragma unroll
        for (int c = 0; c < 8; ++c)
          asm volatile("{\n.reg .pred p;\nsetp.lt.u32 p, %2, %3;\n@p st.shared.f32 [%0], %1;\n}\n" ::"r"(
                           row_at + (h + c) * 4),
                       "f"(y[c]), "r"((uint32_t)(h + c)), "r"(C)
                       : "memory");
      }
      __syncwarp();
      if (P.out_half)
        write(reinterpret_cast<__half *>(out), rowbuf, C, oi, good, lane, P.narrow != 0);
      else
        write(reinterpret_cast<float *>(out), rowbuf, C, oi, good, lane, P.narrow != 0);
      __syncwarp();  // the next tile's rows overwrite the buffer
    }
  }

  static constexpr bool kRowBuffer = H == 128;

  // The roles other than the producers.
  __device__ __forceinline__ void consume(void *out) const {
    if (warp >= kWarpM) {
      const int m = warp - kWarpM;
      if (m < NE)
        issuer(m);
      else if (m == 2)
        loader();
      else if (m == 3)
        dispatcher();
    } else if (warp >= kWarpW) {
      writer(out);
    } else {
      converter((warp - kWarpE) >> 2);
    }
  }
};

// One element of a packed bias block: part j (0 .. kBiasParts - 1) of the bias
// split into values of type T that, times their columns' powers of two, add up to
// it.  An infinite or NaN part stands alone.
template <typename T>
__device__ __forceinline__ T bias_part(float b, uint32_t j) {
  for (uint32_t i = 0;; ++i) {
    const int e = bias_scale(!std::is_same<T, __half>::value, i);
    const T h = T(ldexpf(b, -e));
    if (i == j) return h;
    if (!isfinite((float)h)) return T(0.0f);
    b -= ldexpf((float)h, e);
  }
}

}  // namespace

// The launch arguments that both decodes derive alike.
inline PipeArgs pipe_args(const uint8_t *img, size_t stride, uint32_t k1, uint32_t hidden, uint32_t layers, uint32_t ns,
                          uint32_t producers, uint32_t stages, uint32_t ngrids, uint32_t decoders, uint32_t out_dim, uint32_t out_half,
                          const void *out, size_t n) {
  PipeArgs P{};
  P.img = img;
  P.img_stride = stride;
  P.img_bytes = (uint32_t)pipe_image_bytes(k1, hidden, layers);
  P.ns = ns;
  P.stages = stages;
  P.k1 = k1;
  P.layers = layers;
  P.out_dim = out_dim;
  P.out_half = out_half;
  // vector row stores need 8 channels and a base aligned to the row: 32 bytes
  // (fp32) or 16 (fp16)
  P.vector_rows = out_dim == 8 && ((uintptr_t)out & (out_half ? 15 : 31)) == 0;
  P.narrow = (unsigned long long)n * out_dim < 0xFFFFFFFFull;
  P.sm = PipeSmem::plan(P.img_bytes, ns, producers, ngrids, decoders, out_dim, hidden == 128 && !P.vector_rows);
  return P;
}

}  // namespace ntc
