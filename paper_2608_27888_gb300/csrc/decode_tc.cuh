// The decode of the standard shape (two 8-channel latent grids -> two hidden
// layers of 64 or 128 with ReLU) on the tensor-core pipeline of
// decode_pipe.cuh: its producers, its kernel and its launch.
//
// Shared-memory B operands use the no-swizzle K-major canonical layout: 8-row
// x 16-byte core matrices, K-adjacent core matrices 128 B apart (LBO), 8-row
// groups K*16 B apart (SBO).
//
// This header holds the kernel template; decode_tc.cu instantiates the
// production kernels and decode_tc_debug.cu the debug ones (DBG), in their own
// translation units.
#pragma once

#include "decode_pipe.cuh"

namespace ntc {

constexpr int kTcKA = kInDim + 16;  // K of layer 1's weight image: 16 features + the bias K step

namespace {

// Latent taps of one query from one mip, loaded ahead of use: 2 levels x 4
// taps; a mip blend factor is folded into the weights.
struct Taps {
  static constexpr int N = 8;
  uint4 raw[N];
  float w[N];
};

// Mip selection of one query row, kept between the two fetch phases of a
// kernel that may blend mips.
struct MipPick {
  int lo = 0;
  float t = 0.0f;
};

// One axis of the tap addressing, fp32 round-to-nearest with no contraction
// (the same operations, in the same order, as the reference addressing).
// WRAP: c is finite and the texel pair wraps at the edge; clamp: both texels
// are clamped into [0, n-1].
template <bool WRAP>
__device__ __forceinline__ void axis_pair(float c, uint32_t n, uint32_t &i0, uint32_t &i1, float &frac) {
  const float x = WRAP ? __fsub_rn(__fmul_rn(__fsub_rn(c, floorf(c)), (float)n), 0.5f)
                       : __fsub_rn(__fmul_rn(c, (float)n), 0.5f);
  const float x0f = floorf(x);
  frac = __fsub_rn(x, x0f);
  if (WRAP) {
    const int x0 = (int)x0f;  // in [-1, n-1]
    i0 = x0 < 0 ? n - 1 : (uint32_t)x0;
    const uint32_t a1 = (uint32_t)(x0 + 1);
    i1 = a1 == n ? 0u : a1;
  } else {
    const int x0 = (int)fminf(fmaxf(x0f, -1.0f), (float)n);
    i0 = (uint32_t)min(max(x0, 0), (int)n - 1);
    i1 = (uint32_t)min(x0 + 1, (int)n - 1);
  }
}

// Both texels of one bilinear row from the row-pair copy: one 32-byte load.
struct alignas(32) TexelPair {
  uint4 a, b;
};
__device__ __forceinline__ void ld_pair(const TexelPair *p, uint4 &a, uint4 &b) {
  asm volatile("ld.global.nc.v8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(a.x), "=r"(a.y), "=r"(a.z), "=r"(a.w), "=r"(b.x), "=r"(b.y), "=r"(b.z), "=r"(b.w)
               : "l"(p));
}

// The texel coordinates one grid fetch used (kept only by the debug build).
struct TapIdx {
  uint32_t i0, i1, j0, j1;
};

// Issue the tap loads of one grid (taps 00, 10 from row j0; 01, 11 from row
// j1) and compute their bilinear weights, scaled by sc.  In-grid offsets are
// 32-bit (a grid holds fewer than 2^32 texels).  Clamp mode at an edge has
// x0 = x1, while the pair at x0 holds x0 and its right neighbour: the whole
// row weight then goes to the first texel.  DBG: also report the coordinates.
template <bool WRAP, bool DBG = false>
__device__ __forceinline__ void grid_fetch(const uint4 *pair, const GridDesc &g, float u, float v, float sc,
                                           uint4 *raw, float *w, TapIdx *ti = nullptr) {
  uint32_t i0, i1, j0, j1;
  float fx, fy;
  axis_pair<WRAP>(u, g.W, i0, i1, fx);
  axis_pair<WRAP>(v, g.H, j0, j1, fy);
  if (DBG) *ti = TapIdx{i0, i1, j0, j1};
  const TexelPair *p = reinterpret_cast<const TexelPair *>(pair) + g.base;
  ld_pair(p + (j0 * g.W + i0), raw[0], raw[1]);
  ld_pair(p + (j1 * g.W + i0), raw[2], raw[3]);
  const float ax = __fsub_rn(1.0f, fx), ay = __fsub_rn(1.0f, fy);
  float w00 = __fmul_rn(ax, ay), w10 = __fmul_rn(fx, ay), w01 = __fmul_rn(ax, fy), w11 = __fmul_rn(fx, fy);
  if (!WRAP && i1 == i0) {
    w00 = __fadd_rn(w00, w10);
    w01 = __fadd_rn(w01, w11);
    w10 = w11 = 0.0f;
  }
  w[0] = w00 * sc;
  w[1] = w10 * sc;
  w[2] = w01 * sc;
  w[3] = w11 * sc;
}

// All tap loads of one query from mip lo, issued before any is consumed.  A
// row that is not good (padding, bad set id or UV, bad bucket) fetches texel
// (0, 0) of set 0 instead: no branch and no out-of-range address; its flag
// marks it.  TRI: the kernel may blend mips, so the mip is selected per row
// and mip lo is weighted by 1 - t; otherwise every grid has one mip.
template <bool TRI, bool WRAP, bool DBG = false>
__device__ __forceinline__ void issue_taps(const Assets &A, const GridDesc *grids, const ntc_query &q,
                                           bool good, Taps &tp, MipPick &mp, TapIdx *ti = nullptr) {
  const uint32_t sid = good ? q.set_id : 0u;
  const float u = good ? q.u : 0.0f, v = good ? q.v : 0.0f;
  if (TRI) mp.lo = select_mip(good ? q.lod : 0.0f, A.num_mips, mp.t);
  const uint32_t M = TRI ? A.num_mips : 1u;
  const GridDesc *g = grids + (size_t)sid * kLevels * M;
  const float s = TRI ? __fsub_rn(1.0f, mp.t) : 1.0f;
#pragma unroll
  for (int k = 0; k < kLevels; ++k)
    grid_fetch<WRAP, DBG>(A.pair, g[k * M + mp.lo], u, v, s, tp.raw + 4 * k, tp.w + 4 * k, DBG ? ti + k : nullptr);
}

// The second phase of a mip blend, one level at a time (fewer registers live
// than a whole query's taps): the taps of level k at mip lo + 1, weighted by
// t, for the rows with t > 0 (the others load nothing and get zero weights, so
// their accumulation is unchanged).
template <bool WRAP, bool DBG = false>
__device__ __forceinline__ void issue_level_hi(const Assets &A, const GridDesc *grids, const ntc_query &q,
                                               bool good, const MipPick &mp, int k, uint4 (&raw)[4],
                                               float (&w)[4], TapIdx *ti = nullptr) {
  if (good && mp.t > 0.0f) {
    const uint32_t M = A.num_mips;
    grid_fetch<WRAP, DBG>(A.pair, grids[((size_t)q.set_id * kLevels + k) * M + mp.lo + 1], q.u, q.v, mp.t, raw, w,
                          ti);
  } else {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      w[i] = 0.0f;
      raw[i] = make_uint4(0, 0, 0, 0);
    }
  }
}

// acc[c/2] += w * tap[c] over the 8 channels of one tap, in packed fp16 pairs
// (the latents' own type; hfma2, the first tap multiplies): the feature row
// becomes the fp16/bf16 A operand, so the blend needs no fp32 conversions.
template <bool FIRST>
__device__ __forceinline__ void accum_tap_x2(__half2 (&acc)[4], uint4 raw, float w) {
  const __half2 ww = __float2half2_rn(w);
  const __half2 *h = reinterpret_cast<const __half2 *>(&raw);
#pragma unroll
  for (int p = 0; p < 4; ++p) acc[p] = FIRST ? __hmul2(ww, h[p]) : __hfma2(ww, h[p], acc[p]);
}

// Feature accumulation: acc[k][c/2] over the 8 channels of level k, all taps
// of mip lo first (FIRST: the first tap multiplies), then those of mip lo + 1.
template <bool FIRST>
__device__ __forceinline__ void accum_taps(const Taps &tp, __half2 (&acc)[kLevels][4]) {
#pragma unroll
  for (int k = 0; k < kLevels; ++k) {
    accum_tap_x2<FIRST>(acc[k], tp.raw[k * 4], tp.w[k * 4]);
#pragma unroll
    for (int p = 1; p < 4; ++p) accum_tap_x2<false>(acc[k], tp.raw[k * 4 + p], tp.w[k * 4 + p]);
  }
}

template <bool BF16>
__device__ __forceinline__ void pack_row(const __half2 (&acc)[kLevels][4], uint32_t (&packed)[8]) {
#pragma unroll
  for (int k = 0; k < kLevels; ++k)
#pragma unroll
    for (int p = 0; p < 4; ++p) {
      if (BF16) {
        const float2 x = __half22float2(acc[k][p]);
        packed[k * 4 + p] = pack<true>(x.x, x.y);
      } else {
        packed[k * 4 + p] = *reinterpret_cast<const uint32_t *>(&acc[k][p]);
      }
    }
}

// How the standard shape fills the pipeline: four producer warpgroups and two
// converters; four tile slots at H = 64 and two at H = 128, where tensor memory
// holds no more.  IMAGES weight images in shared memory (16.5 KB at H = 64,
// 48.5 KB at H = 128).
template <int H>
struct TmShape {
  static constexpr int NP = 4, NE = 2, T = H == 64 ? 4 : 2, IMAGES = T;
};
template <int H, bool BF16>
using TmPipe = Pipe<H, BF16, TmShape<H>::NP, TmShape<H>::NE, TmShape<H>::T, kInDim, 2>;

// The producers of the standard shape.  A thread builds one row of a
// tile: bilinear taps of both grids (the same fp32 operations as the reference
// addressing), each bilinear row one 32-byte load from the row-pair copy of the
// latents, blended in packed fp16 (the latents' own type).
// DBG (a separate instantiation, for tests): every producer also records the
// row it built -- texel indices, the 16 bytes blended for each tap, their
// weights, the mip pick and the packed feature row -- in dbg[output row].
template <int H, bool BF16, bool TRI, bool WRAP, bool DBG>
__device__ __forceinline__ void produce_tm(const TmPipe<H, BF16> &pipe, const Assets &A, const Buckets &B,
                                           const GridDesc *grids, void *out, unsigned long long *err,
                                           ntc_debug_row *dbg) {
  constexpr uint32_t NP = TmShape<H>::NP;
  const uint32_t K = pipe.K;
  const uint32_t p = (uint32_t)pipe.warp >> 2, row = threadIdx.x & 127;  // tiles p, p + NP, ...
  const int lane = pipe.lane;
  typename TmPipe<H, BF16>::Rows rows(pipe, B, p);
  for (uint32_t k = p, j = 0; k < K && !pipe.wait.stopped(); k += NP, ++j) {
    const ntc_query q = rows.record();
    const uint32_t oi = rows.oi;
    const bool valid = oi != kNoRow;
    const bool good = valid && !query_bad(A, q);
    rows.look_ahead(pipe, k, rows.oi);
    Taps taps;
    MipPick mp;
    TapIdx ti[kLevels];
    issue_taps<TRI, WRAP, DBG>(A, grids, q, good, taps, mp, ti);
    // the record of a debug build: texel (i, j) of grid (set, level, mip) is
    // texel base + j * W + i of the caller's latents
    auto record = [&](int lv, int slot, const uint4 *raw, const float *w, const TapIdx &x) {
      ntc_debug_row &r = dbg[oi];
      const GridDesc gl = A.grids[((size_t)q.set_id * kLevels + lv) * A.num_mips + mp.lo + slot];
      const unsigned long long r0 = gl.base + (unsigned long long)x.j0 * gl.W;
      const unsigned long long r1 = gl.base + (unsigned long long)x.j1 * gl.W;
      r.idx[lv][slot][0] = r0 + x.i0;
      r.idx[lv][slot][1] = r0 + x.i1;
      r.idx[lv][slot][2] = r1 + x.i0;
      r.idx[lv][slot][3] = r1 + x.i1;
#pragma unroll
      for (int p = 0; p < 4; ++p) {
        r.raw[lv][slot][p][0] = raw[p].x;
        r.raw[lv][slot][p][1] = raw[p].y;
        r.raw[lv][slot][p][2] = raw[p].z;
        r.raw[lv][slot][p][3] = raw[p].w;
        r.w[lv][slot][p] = w[p];
      }
    };
    if (DBG && good) {
      dbg[oi].t = mp.t;
      dbg[oi].lo = (uint32_t)mp.lo;
#pragma unroll
      for (int lv = 0; lv < kLevels; ++lv) record(lv, 0, taps.raw + 4 * lv, taps.w + 4 * lv, ti[lv]);
    }
    // bad rows (set id out of range, non-finite UV, or the bad bucket) decode to NaN
    const bool bad = valid && !good;
    const uint32_t badm = __ballot_sync(0xFFFFFFFFu, bad);
    if (badm && lane == __ffs(badm) - 1) atomicAdd(err, (unsigned long long)__popc(badm));
    if (bad) put_nan_row(out, oi, pipe.P.out_dim, pipe.P.out_half);
    __half2 acc[kLevels][4];
    accum_taps<true>(taps, acc);
    if (TRI && __any_sync(0xFFFFFFFFu, good && mp.t > 0.0f)) {  // some row blends two mips
      uint4 raw[kLevels][4];  // both levels' loads in flight
      float w[kLevels][4];
      TapIdx th[kLevels];
#pragma unroll
      for (int lv = 0; lv < kLevels; ++lv) issue_level_hi<WRAP, DBG>(A, grids, q, good, mp, lv, raw[lv], w[lv], th + lv);
#pragma unroll
      for (int lv = 0; lv < kLevels; ++lv) {
        if (DBG && good && mp.t > 0.0f) record(lv, 1, raw[lv], w[lv], th[lv]);
#pragma unroll
        for (int t = 0; t < 4; ++t) accum_tap_x2<false>(acc[lv], raw[lv][t], w[lv][t]);
      }
    }
    uint32_t a[8];
    pack_row<BF16>(acc, a);
    if (DBG && good)
#pragma unroll
      for (int i = 0; i < 8; ++i) dbg[oi].feat[i] = a[i];
    if (k < pipe.Kg) pipe.hand_over(p, j, k, row, a, good ? oi : kNoRow);  // (a bad bucket's rows end here)
  }
}

template <int H, bool BF16, bool TRI, bool WRAP, bool DBG>
__global__ void __launch_bounds__(TmPipe<H, BF16>::kThreads, 1)
    k_decode_tm(Assets A, Buckets B, const __grid_constant__ PipeArgs P, void *out, unsigned long long *err,
                unsigned int *status, ntc_debug_row *dbg) {
  extern __shared__ __align__(128) uint8_t smem[];
  const GridDesc *grids = A.pgrids;  // grid bases in the row-pair copy
  const TmPipe<H, BF16> pipe(P, smem, B, A.num_decoders, status, grids, A.num_sets * kLevels * A.num_mips);
  if (pipe.warp < pipe.kWarpE)
    produce_tm<H, BF16, TRI, WRAP, DBG>(pipe, A, B, grids, out, err, dbg);
  else
    pipe.consume(out);
  pipe.end();
}

template <int H, bool BF16, bool TRI, bool WRAP, bool DBG>
cudaError_t launch_tm_t(const Assets &A, const WeightImages &W, const Buckets &B, size_t n, void *out,
                        unsigned long long *err, unsigned int *status, int num_sms, cudaStream_t st,
                        ntc_debug_row *dbg) {
  using S = TmShape<H>;
  const PipeArgs P = pipe_args(W.tc, W.tc_stride, kInDim, H, 2, S::IMAGES, S::NP, S::NP, A.num_sets * kLevels * A.num_mips,
                               A.num_decoders, W.out_dim, W.out_half, out, n);
  static_assert(pipe_columns(H, S::T, kInDim, S::NP) <= 512, "tensor memory plan exceeds 512 columns");
  const auto kernel = k_decode_tm<H, BF16, TRI, WRAP, DBG>;
  static PerDevice attr;
  cudaError_t e = attr.once([&]() {
    const PipeSmem most = PipeSmem::plan(P.img_bytes, S::IMAGES, S::NP, kSmemGrids, kSmemTileTable - 2, 16, true);
    return allow_smem((const void *)kernel, most.total);
  });
  if (e != cudaSuccess) return e;
  const size_t max_tiles = (n + kTile - 1) / kTile + A.num_decoders + 1;
  size_t grid = (size_t)num_sms;
  if (grid > max_tiles) grid = max_tiles;
  // launched as a programmatic dependent of the bucketing: its prologue overlaps
  // the end of k_place
  e = launch_pdl_l1(kernel, dim3((unsigned)grid), dim3(TmPipe<H, BF16>::kThreads), P.sm.total, st, A, B, P, out, err,
                    status, dbg);
  if (e != cudaSuccess) return e;
  return cudaGetLastError();
}

}  // namespace

// Every (H, precision, trilinear, address mode) shape of the standard decode,
// dispatched at run time.
template <bool DBG>
cudaError_t dispatch_tm(const Assets &A, const WeightImages &W, const Buckets &B, size_t n, void *out,
                        unsigned long long *err, unsigned int *status, bool bf16, int num_sms, cudaStream_t st,
                        ntc_debug_row *dbg) {
  const bool tri = A.num_mips > 1, wrap = A.address_mode == 0;
#define NTC_TM(H, BF, TRI, WRAP) return launch_tm_t<H, BF, TRI, WRAP, DBG>(A, W, B, n, out, err, status, num_sms, st, dbg)
#define NTC_TM_H(H)                             \
  do {                                          \
    if (bf16) {                                 \
      if (tri && wrap) NTC_TM(H, true, true, true);   \
      if (tri) NTC_TM(H, true, true, false);    \
      if (wrap) NTC_TM(H, true, false, true);   \
      NTC_TM(H, true, false, false);            \
    }                                           \
    if (tri && wrap) NTC_TM(H, false, true, true);    \
    if (tri) NTC_TM(H, false, true, false);     \
    if (wrap) NTC_TM(H, false, false, true);    \
    NTC_TM(H, false, false, false);             \
  } while (0)
  if (W.hidden == 64) NTC_TM_H(64);
  NTC_TM_H(128);
#undef NTC_TM_H
#undef NTC_TM
}

}  // namespace ntc
