// Softmax attention on fp32 tensors at head_dim 64 (Eq. 1, full and windowed, with prefix tokens): fp32
// multiply-adds throughout, register-tiled.
//
// What bounds it: the FMA pipes (4 * 64 flop per query-key pair; 128 multiply-adds per clock and SM).  A warp
// owns 16 query rows and walks tiles of 64 keys (short rows of keys: 32); a lane owns 8 rows x 4 keys of the scores (keys lane % 16 + 16 j)
// and 8 rows x 4 channels of the output.  Multiply-adds are packed pairs (fma.rn.f32x2: even and odd channels
// in QK^T, two neighbouring rows in PV), fed by 128-bit shared-memory loads: 12 loads per 64 packed
// multiply-adds, three quarters of what the shared-memory port could deliver.  The rows of a
// warp see all keys of a tile inside that warp: row maxima are 16-lane shuffles and the probabilities pass from the
// score layout to the PV layout through the warp's own shared memory, without a CTA barrier.  They are kept by key, so that
// a load gives pairs of rows and a value is doubled once for eight rows (kept by row, with pairs of channels, every
// probability had to be doubled: 98 us where this takes 93).
//
// A CTA is R row warps x G key groups: group g takes the key tiles g, g + G, ... through its own buffer (K, then V in its
// place: with three CTAs on an SM the others compute while one waits for a copy), and the groups' partial softmaxes are
// merged at the end.
//
// It serves what does not fill the chip with its row tiles, rows of up to 64 keys, short rows of queries and the prefix queries of windows; the rest goes to the
// tensor cores (attn_f32_tc.cu; the line between the two: launch_attn_f32).  Measured (6 heads, 16 x 16 tokens; the kernel of one warp
// per query row, which serves other head dims and windows of at most eight tokens, in brackets): full attention 8 us (63).  Where it fills the chip it
// runs at 35 to 41 TFLOP/s of the 73 that a loop of nothing but multiply-adds reaches: one of three instructions is not a
// multiply-add, and the registers leave room for three warps per scheduler.
#include <cooperative_groups.h>

#include <type_traits>

#include "f32_common.cuh"

namespace jv {
namespace {

using namespace f32;

constexpr int kTileKeys = 64;    // keys per tile, but for short rows of keys
// floats of a warp's own buffer: the probabilities of a tile of `keys` keys, then the warp's output
__host__ __device__ constexpr int warp_buf(int keys) { return keys * kLdP > kRowsWarp * kLd ? keys * kLdP : kRowsWarp * kLd; }

template <int R, int G, int kKeys>
constexpr size_t smem_bytes() {
  return ((size_t)(R * kRowsWarp + G * kKeys) * kLd + R * G * warp_buf(kKeys)) * sizeof(float);
}

// kPrefix: the launch serves the P prefix queries (keys: all tokens) instead of the windows, by clusters of blocks along x that
// share the keys of a row tile and merge their partial softmaxes through distributed shared memory.
// kKeys: keys per tile, 64, or 32 where that leaves no group without one
template <int R, int G, int kKeys, bool kPrefix>
__global__ void __launch_bounds__(32 * R * G, G == 2 ? 3 : G == 4 ? 2 : 1)  // what shared memory leaves room for
attn_f32_kernel(const float* __restrict__ q, const float* __restrict__ k, const float* __restrict__ v, float* __restrict__ o,
                const int* status, int Hg, int Wg, int P, int wh, int ww, int nwx, bool overlap, float scale) {
  namespace cg = cooperative_groups;
  constexpr int kWarpBuf = warp_buf(kKeys);
  extern __shared__ __align__(16) float smem_f[];
  float* qs = smem_f;                                        // [16 R][kLd]
  float* ps = qs + R * kRowsWarp * kLd;                      // [R G warps]: probabilities [kKeys][kLdP], then the warp's output [16][kLd]
  float* ks = ps + R * G * kWarpBuf;                         // [G][kKeys][kLd]: the group's K tile, then its V tile
  // overlap: the launch ahead is that of the prefix queries (it has waited for what came before it); waited for at the end
  if (!overlap) griddep_wait();
  griddep_launch_dependents();
  // an earlier kernel gave up, and the windows' kernel looks at the word, too: o stays as it is (status null: that one does not)
  const bool gave_up = kPrefix && status && *reinterpret_cast<const volatile int*>(status) != 0;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, tx = lane & 15, ty = lane >> 4;
  const int grp = warp / R, rw = warp % R;                   // key group, row warp
  const int N = P + Hg * Wg;
  const int nsplit = kPrefix ? (int)cg::this_cluster().num_blocks() : 1, split = kPrefix ? (int)cg::this_cluster().block_rank() : 0;
  const int wy = blockIdx.y / nwx, wx = blockIdx.y % nwx;
  const int y0 = kPrefix ? 0 : wy * wh, x0 = kPrefix ? 0 : wx * ww;
  const int vh = min(wh, Hg - y0), vw = min(ww, Wg - x0);    // valid extent of this window
  const int nq = kPrefix ? P : vh * vw;                  // query rows; keys: prefix tokens, then the window's own
  const int cnt = kPrefix ? N : P + vh * vw;
  const int row0 = blockIdx.x / nsplit * (R * kRowsWarp);
  if (row0 >= nq) return;                                    // beyond a small edge window
  const size_t base = (size_t)blockIdx.z * N * kDim;
  const bool dense = kPrefix || vw == Wg;                // consecutive keys are consecutive tokens
  auto key_token = [&](int c) -> int {
    if (c < P) return c;
    if (dense) return kPrefix ? c : c + y0 * Wg;
    const int g = c - P, y = g / vw;
    return P + (y0 + y) * Wg + x0 + (g - y * vw);
  };

  // the group's tile t of K or V: warp rw copies rows [64 / R * rw, + 64 / R), half a warp per row
  auto load_tile = [&](float* dst, const float* src, int t) {
    constexpr int kOwn = kKeys / R;                          // rows of this warp
    int tok[(kOwn + 31) / 32];
#pragma unroll
    for (int i = 0; i < (kOwn + 31) / 32; ++i) {
      const int c = t * kKeys + rw * kOwn + 32 * i + (kOwn < 32 ? lane % kOwn : lane);
      tok[i] = c < cnt ? key_token(c) : -1;
    }
#pragma unroll
    for (int j = 0; j < kOwn / 2; ++j) {
      const int r = 2 * j + ty;
      const int tk = __shfl_sync(0xffffffffu, tok[(2 * j) / 32], r & 31);
      copy16(dst + (rw * kOwn + r) * kLd + 4 * tx, src + base + (size_t)max(tk, 0) * kDim + 4 * tx, tk >= 0);
    }
    copy_commit();
  };
  auto group_sync = [&]() {
    if (R == 1) __syncwarp();
    else asm volatile("bar.sync %0, %1;" ::"r"(1 + grp), "n"(32 * R) : "memory");
  };

  float* kg = ks + grp * kKeys * kLd;
  float* pw = ps + warp * kWarpBuf;
  const int ntiles = (cnt + kKeys - 1) / kKeys;
  const int first = split * G + grp, stride = nsplit * G;

  if (grp == 0) {                                            // Q: group 0 copies the CTA's rows
    const int mine = row0 + rw * kRowsWarp + (lane & 15);
    const int tok = mine < nq ? key_token(kPrefix ? mine : P + mine) : -1;
#pragma unroll
    for (int j = 0; j < kRowsWarp / 2; ++j) {
      const int r = 2 * j + ty, tk = __shfl_sync(0xffffffffu, tok, r);
      copy16(qs + (rw * kRowsWarp + r) * kLd + 4 * tx, q + base + (size_t)max(tk, 0) * kDim + 4 * tx, tk >= 0);
    }
  }
  if (first < ntiles) load_tile(kg, k, first);                   // (one copy group with Q)
  else copy_commit();
  if (G > 1) {                                               // Q comes from group 0: everybody waits for it once
    copy_wait<0>();
    __syncthreads();
  }

  const float* qr = qs + (rw * kRowsWarp + ty * 8) * kLd;
  RowTile<kKeys> x;
  for (int t = first; t < ntiles; t += stride) {
    copy_wait<0>();                                          // K of this tile
    group_sync();
    x.scores(qr, kg, tx);
    group_sync();                                            // the group is done with K
    load_tile(kg, v, t);                                     // V, under the softmax

    x.softmax(cnt - t * kKeys, scale, pw, tx, ty);
    copy_wait<0>();                                          // V of this tile
    group_sync();                                            // (also orders the warp's own probabilities)
    x.values(kg, pw, tx, ty);
    group_sync();                                            // the group is done with V (and the warp with its P)
    if (t + stride < ntiles) load_tile(kg, k, t + stride);
  }

  x.finish();
  // Merge the groups through the warps' own buffers: output channels 0..63 of a row, then its maximum and sum.
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    float* dst = pw + (ty * 8 + i) * kLd;
    *reinterpret_cast<float4*>(dst + 4 * tx) = x.row(i);
    if (tx == 0) {
      dst[64] = x.m[i];
      dst[65] = x.l[i];
    }
  }
  __syncthreads();
  // n <= kMost partial softmaxes of a row -> maximum, sum and this lane's four channels.  Unrolled, so that all of them are on their way at once.
  auto combine = [&](auto most, int n, auto&& src_of, float& M, float& L) -> float4 {
    constexpr int kMost = decltype(most)::value;
    float m[kMost];
    M = -INFINITY;
#pragma unroll
    for (int i = 0; i < kMost; ++i) {
      m[i] = i < n ? src_of(i)[64] : -INFINITY;
      M = fmaxf(M, m[i]);
    }
    const float ref = M == -INFINITY ? 0.f : M;
    L = 0.f;
    float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int i = 0; i < kMost; ++i) {
      if (i >= n) continue;
      const float* src = src_of(i);
      const float f = expf(m[i] - ref);                                // a source without a key of weight: exp(-inf) = 0
      const float4 y = *reinterpret_cast<const float4*>(src + 4 * tx);
      L = fmaf(src[65], f, L);
      x.x = fmaf(y.x, f, x.x);
      x.y = fmaf(y.y, f, x.y);
      x.z = fmaf(y.z, f, x.z);
      x.w = fmaf(y.w, f, x.w);
    }
    return x;
  };
  auto store = [&](int row, const float4& x, float L) {
    const float inv = 1.f / L;
    const int tok = key_token(kPrefix ? row : P + row);
    if (!gave_up) *reinterpret_cast<float4*>(o + base + (size_t)tok * kDim + 4 * tx) = make_float4(x.x * inv, x.y * inv, x.z * inv, x.w * inv);
  };
  constexpr int kOwnRows = kRowsWarp / G;                    // rows of row warp rw that this warp writes out
#pragma unroll
  for (int j = 0; j < kOwnRows / 2; ++j) {
    const int r = grp * kOwnRows + 2 * j + ty, row = row0 + rw * kRowsWarp + r;
    if (row < nq) {
      float M, L;
      const float4 x = combine(std::integral_constant<int, G>(), G, [&](int g) { return ps + (g * R + rw) * kWarpBuf + r * kLd; }, M, L);
      if (nsplit == 1) {
        store(row, x, L);
      } else {                                               // this block's share, over Q
        float* dst = qs + (rw * kRowsWarp + r) * kLd;
        *reinterpret_cast<float4*>(dst + 4 * tx) = x;
        if (tx == 0) {
          dst[64] = M;
          dst[65] = L;
        }
      }
    }
  }
  if (kPrefix && nsplit > 1) {
    cg::cluster_group cluster = cg::this_cluster();
    cluster.sync();
    for (int r = split + nsplit * (2 * warp + ty); r < R * kRowsWarp; r += 2 * R * G * nsplit)   // (uniform over 16 lanes)
      if (row0 + r < nq) {
        float M, L;
        const float4 x = combine(std::integral_constant<int, 8>(), nsplit, [&](int i) { return cluster.map_shared_rank(qs, i) + r * kLd; }, M, L);
        store(row0 + r, x, L);
      }
    cluster.sync();                                          // no block leaves while its shared memory may still be read
  }
  if (overlap) griddep_wait();
}

template <int R, int G, int kKeys, bool kPrefix>
cudaError_t launch(const AttnArgs& a, int split, const int* status, bool overlap, cudaStream_t st) {   // split: blocks to a cluster (the prefix queries)
  static OncePerDevice opt_in;
  const cudaError_t e = opt_in.run([&] {
    return cudaFuncSetAttribute(attn_f32_kernel<R, G, kKeys, kPrefix>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)smem_bytes<R, G, kKeys>());
  });
  if (e != cudaSuccess) return e;
  const int wh = a.wh < a.Hg ? a.wh : a.Hg, ww = a.ww < a.Wg ? a.ww : a.Wg;
  const int nwx = ceil_div(a.Wg, ww), nwin = nwx * ceil_div(a.Hg, wh);
  const dim3 grid = kPrefix ? dim3(ceil_div(a.P, R * kRowsWarp) * split, 1, a.BH) : dim3(ceil_div(wh * ww, R * kRowsWarp), nwin, a.BH);
  return launch_cluster(true, attn_f32_kernel<R, G, kKeys, kPrefix>, kPrefix ? split : 0, grid, 32 * R * G, smem_bytes<R, G, kKeys>(), st, (const float*)a.q,
                        (const float*)a.k, (const float*)a.v, (float*)a.o, status, a.Hg, a.Wg, a.P, wh, ww, nwx, overlap, a.scale);
}

}  // namespace

bool attn_f32_supported(const AttnArgs& a) { return a.dtype == JV_F32 && a.D == kDim && !a.strided; }

// The P prefix queries go first, with the keys of a row tile split over the four groups of up to eight blocks (their chain is the longest: all
// N keys), two blocks to an SM; the windows' launch overlaps them, as neither reads what the other writes.  One block of four groups / as many as
// the rule gives, us for the call with 16 x 16 windows: 6 heads of 37 x 37, 5 prefix tokens 32.8 / 16.5, 24 of 24 x 24 35.3 / 27.7, 48 of 37 x 37 105.8 / 80.8, 192
// 309 / 309.  More than 16 prefix tokens are several row tiles per head: a second block per SM is worth it only where the groups have more than
// a tile each (6 heads of 20 x 20, 120 prefix tokens, 5 x 5 windows, one / two blocks per SM 16.4 / 19.7, of 24 x 24, 100, 4 x 4 20.7 / 15.8), and where the tiles
// alone give most SMs a block, that one has eight groups (12 heads of 24 x 24, 120, 5 x 5, two of four groups / one of eight 37.0 / 35.2; of 32 x 32 54.2 / 49.1).
//
// Windows and sequences go to the tensor cores (attn_f32_tc.cu) where they fill the chip with row tiles of this kernel.  That one's blocks
// take 128 rows, or two windows of up to 64, and start slowly: 10 us for two tiles of keys, 12 for four, where this one takes 7 to 8 as long as every SM
// has one block.  This / that one, us:
//   up to 64 keys: always here.  96 heads of 64 tokens 7.6 / 8.4, 384 17.8 / 17.8; 8 x 8 windows, 48 heads of 32 x 32 32.0 / 31.7, 192 of 20 x 20
//     48.0 / 64.4; 7 x 7, 96 of 24 x 24 45.3 / 53.5 (6 x 6, 48 of 24 x 24 30.2 / 28.1);
//   up to 128: 192 heads of 100 28.5 / 19.7, 48 of 100 11.1 / 9.5; of windows (8 x 8, 5 prefix tokens) 24 heads of 16 x 16 12.9 / 14.3, 12 of 20 x 20
//     12.7 / 13.4, 24 of 24 x 24 24.6 / 23.4, 48 of 16 x 16 21.5 / 15.1, 192 of 20 x 20 88 / 91;
//   up to 256: 6 heads of 256 8.2 / 12.5, 12 of 256 11.6 / 12.6, 24 of 256 17.6 / 12.5; 16 x 16 windows, 6 heads of 24 x 24 11.8 / 12.7;
//   more: 6 heads of 300 12.7 / 14.0, 6 of 400 19.0 / 15.6, 12 of 1024 93 / 27.9.
// Rows of at most 32 queries stay here (a tile there would be three quarters empty): 4 x 4 windows, 48 heads of 32 x 32 72 / 87.
//
// Here, 32 rows x 2 groups per CTA (three on an SM) or 16 rows x 4 groups (two): the second halves the chain of a CTA, the first is faster
// where both fill the chip several times and its 32 rows are filled.  More than 128 keys and 17 to 32 queries, 16 x 4 / 32 x 2 (5 x 5 windows, 120 prefix tokens): 6 heads of
// 16 x 16 12.5 / 20.8, 12 of 24 x 24 35.1 / 39.5, 12 of 32 x 32 55.1 / 48.9, 192 of 24 x 24 392 / 347.  Up to 128, 24 heads of 16 x 16, 8 x 8 windows,
// 5 prefix tokens 18.2 / 12.9; 4 x 4 windows, 100, 96 heads of 24 x 24 129 / 159.
// Short rows of keys (up to 64, 128 and 256) are cut into tiles of 32, so that two, four or eight groups have one each and a
// CTA's chain is half as long.  Tiles of 64 / of 32, us: 6 heads of 64 tokens 7.5 / 5.4, of 128 8.1 / 5.3, 24 of 128 8.3 / 7.4, 6 of 200 8.0 / 7.4, of 256 8.3 /
// 8.2; 8 x 8 windows, 6 heads of 16 x 16 8.2 / 5.8, 4 x 4, 24 of 32 x 32 40 / 27.  Eight groups take an SM: only where every row tile gets one (12 heads
// of 256 tokens 11.7 / 14.8).
// Windows of at most eight tokens leave most of a 32 x 64 tile of scores empty: the kernel of one warp per query row, eight to a block, is the
// better one.  This one / that one, 96 heads of 32 x 32 tokens: 2 x 2 windows 484 / 270 us, 2 x 4 256 / 148, 3 x 3 245 / 254; 12 heads of 64 x 64, 2 x 2
// 235 / 135.  With prefix tokens, whose queries stay here: as long as a window's keys and they are one tile of that kernel, and the windows fill
// the chip several times (it does not overlap the prefix queries): 12 heads of 64 x 64, 2 x 2, 5 prefix tokens 299 / 207, 40: 301 / 337; 6 heads of
// 16 x 16, 1 x 1 36.7 / 30.8, 1 x 2 20.4 / 23.3, 2 x 2 11.9 / 18.5; of 37 x 37, 1 x 7 50.5 / 47.1.
cudaError_t launch_attn_f32(const AttnArgs& a, cudaStream_t st) {
  const int wh = a.wh < a.Hg ? a.wh : a.Hg, ww = a.ww < a.Wg ? a.ww : a.Wg;
  const bool prefix = a.P > 0;
  const int64_t sms = device_sm_count(), windows = (int64_t)ceil_div(a.Wg, ww) * ceil_div(a.Hg, wh) * a.BH;
  const int nq = wh * ww, cnt = a.P + nq, key_tiles = ceil_div(cnt, kTileKeys);
  // row tiles of this kernel: small windows at the edges have fewer
  auto row_tiles = [&](int rows) -> int64_t {
    const int ny = a.Hg / wh, nx = a.Wg / ww, eh = a.Hg % wh, ew = a.Wg % ww;
    return a.BH * ((int64_t)ny * nx * ceil_div(nq, rows) + (int64_t)nx * ceil_div(eh * ww, rows) + (int64_t)ny * ceil_div(wh * ew, rows) + ceil_div(eh * ew, rows));
  };
  const int64_t rows16 = row_tiles(kRowsWarp), rows32 = row_tiles(2 * kRowsWarp);
  bool tc = nq > 2 * kRowsWarp && a.scale >= 0x1p-40f && a.scale <= 0x1p40f;   // (else what its terms do not hold of very small or infinite values may count)
  if (cnt <= kTileKeys) tc = false;
  else if (cnt <= 2 * kTileKeys) tc = tc && rows32 > sms && (nq > kTileKeys || rows32 > 2 * sms);
  else tc = tc && rows16 > sms && (key_tiles > 4 || 2 * rows16 > 3 * sms);
  int* status = nullptr;                                   // for the kernels of a call that leave o alone while the word is set: all of them, or none
  if (tc && !(status = device_status_ptr())) return cudaErrorUnknown;
  if (prefix) {
    const int N = a.P + a.Hg * a.Wg;
    const int64_t tiles = (int64_t)ceil_div(a.P, kRowsWarp) * a.BH;
    int split = 1;
    while (split < 8 && split * tiles <= sms && split * 4 * kTileKeys < N &&
           (a.P <= kRowsWarp || 2 * split * tiles <= sms || split * 5 * kTileKeys <= N)) split *= 2;
    const bool eight = a.P > kRowsWarp && 2 * tiles > sms && tiles <= sms;
    const cudaError_t e = eight ? launch<1, 8, kTileKeys, true>(a, 1, status, false, st) : launch<1, 4, kTileKeys, true>(a, split, status, false, st);
    if (e != cudaSuccess) return e;
  }
  if (tc) return launch_attn_f32_tc(a, prefix, status, st);
  if (nq <= 8 && (!prefix || (cnt <= 32 && windows >= 8 * sms))) return launch_attn_generic(a, st, true);
  if (cnt <= kTileKeys) return launch<2, 2, 32, false>(a, 1, nullptr, prefix, st);
  if (cnt <= 2 * kTileKeys && (nq <= kRowsWarp || rows16 <= 2 * sms)) return launch<1, 4, 32, false>(a, 1, nullptr, prefix, st);
  if (cnt <= 4 * kTileKeys && rows16 <= sms) return launch<1, 8, 32, false>(a, 1, nullptr, prefix, st);
  const int64_t rounds2 = (windows * ceil_div(nq, 2 * kRowsWarp) + sms - 1) / sms, rounds1 = (windows * ceil_div(nq, kRowsWarp) + sms - 1) / sms;
  if (cnt > 2 * kTileKeys && (rounds2 <= 2 || 5 * rounds1 <= 9 * rounds2)) return launch<1, 4, kTileKeys, false>(a, 1, nullptr, prefix, st);
  return launch<2, 2, kTileKeys, false>(a, 1, nullptr, prefix, st);
}

}  // namespace jv
