// Softmax attention on fp32 tensors at head_dim 64 (Eq. 1, full and windowed, with prefix tokens): fp32
// multiply-adds throughout, register-tiled.
//
// What bounds it: the FMA pipes (4 * 64 flop per query-key pair; 128 multiply-adds per clock and SM).  A warp
// owns 16 query rows and walks tiles of 64 keys; a lane owns 8 rows x 4 keys of the scores (keys lane % 16 + 16 j)
// and 8 rows x 4 channels of the output.  Multiply-adds are packed pairs (fma.rn.f32x2: even and odd channels
// in QK^T, two neighbouring channels in PV), fed by 128-bit shared-memory loads: 12 loads per 64 packed
// multiply-adds, half of what the shared-memory port could deliver, so the FMA pipes stay the limit.  The rows of a
// warp see all keys of a tile inside that warp: row maxima are 16-lane shuffles and the probabilities pass from the
// score layout to the PV layout through the warp's own shared memory, without a CTA barrier.
//
// A CTA is R row warps x G key groups: group g takes the key tiles g, g + G, ... through its own buffer (K, then V in its
// place: with three CTAs on an SM the others compute while one waits for a copy), and the groups' partial softmaxes are
// merged at the end.
//
// Measured (12 heads, 32 x 32 tokens; the kernel of one warp per query row, which served these calls before and still
// serves other head dims, in brackets): full attention 100 us (729), 16 x 16 windows 31 us (195); 6 heads, 16 x 16
// tokens, full attention 10 us (63).  Full attention runs at 32 TFLOP/s of the 73 that a loop of nothing but multiply-adds
// reaches: two of five instructions are not multiply-adds, and the registers leave room for three warps per scheduler.
#include "f32_common.cuh"

namespace jv {
namespace {

using namespace f32;

constexpr int kDim = 64;
constexpr int kKeys = 64;        // keys per tile
constexpr int kRowsWarp = 16;    // query rows per warp
constexpr int kLd = 68;          // floats per shared-memory row: 16-byte reads of 8 consecutive rows touch all banks

template <int R, int G>
constexpr size_t smem_bytes() {
  return (size_t)(R * kRowsWarp + R * G * kRowsWarp + G * kKeys) * kLd * sizeof(float);
}

// prefix_rows: the launch serves the P prefix queries (keys: all tokens) instead of the windows.
template <int R, int G>
__global__ void __launch_bounds__(32 * R * G, 3)
attn_f32_kernel(const float* __restrict__ q, const float* __restrict__ k, const float* __restrict__ v, float* __restrict__ o,
                int Hg, int Wg, int P, int wh, int ww, int nwx, bool prefix_rows, bool overlap, float scale) {
  extern __shared__ __align__(16) float smem_f[];
  float* qs = smem_f;                                        // [16 R][kLd]
  float* ps = qs + R * kRowsWarp * kLd;                      // [R G warps][16][kLd]: probabilities, then the warp's output
  float* ks = ps + R * G * kRowsWarp * kLd;                  // [G][64][kLd]: the group's K tile, then its V tile
  // overlap: the launch ahead is that of the prefix queries (it has waited for what came before it); waited for at the end
  if (!overlap) griddep_wait();
  griddep_launch_dependents();

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, tx = lane & 15, ty = lane >> 4;
  const int grp = warp / R, rw = warp % R;                   // key group, row warp
  const int N = P + Hg * Wg;
  const int wy = blockIdx.y / nwx, wx = blockIdx.y % nwx;
  const int y0 = prefix_rows ? 0 : wy * wh, x0 = prefix_rows ? 0 : wx * ww;
  const int vh = min(wh, Hg - y0), vw = min(ww, Wg - x0);    // valid extent of this window
  const int nq = prefix_rows ? P : vh * vw;                  // query rows; keys: prefix tokens, then the window's own
  const int cnt = prefix_rows ? N : P + vh * vw;
  const int row0 = blockIdx.x * (R * kRowsWarp);
  if (row0 >= nq) return;                                    // beyond a small edge window
  const size_t base = (size_t)blockIdx.z * N * kDim;
  const bool dense = prefix_rows || vw == Wg;                // consecutive keys are consecutive tokens
  auto key_token = [&](int c) -> int {
    if (c < P) return c;
    if (dense) return prefix_rows ? c : c + y0 * Wg;
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
  float* pw = ps + warp * kRowsWarp * kLd;
  const int ntiles = (cnt + kKeys - 1) / kKeys;

  if (grp == 0) {                                            // Q: group 0 copies the CTA's rows
    const int mine = row0 + rw * kRowsWarp + (lane & 15);
    const int tok = mine < nq ? key_token(prefix_rows ? mine : P + mine) : -1;
#pragma unroll
    for (int j = 0; j < kRowsWarp / 2; ++j) {
      const int r = 2 * j + ty, tk = __shfl_sync(0xffffffffu, tok, r);
      copy16(qs + (rw * kRowsWarp + r) * kLd + 4 * tx, q + base + (size_t)max(tk, 0) * kDim + 4 * tx, tk >= 0);
    }
  }
  if (grp < ntiles) load_tile(kg, k, grp);                   // (one copy group with Q)
  else copy_commit();
  if (G > 1) {                                               // Q comes from group 0: everybody waits for it once
    copy_wait<0>();
    __syncthreads();
  }

  const float* qr = qs + (rw * kRowsWarp + ty * 8) * kLd;
  float m[8], l[8];
  f32x2 acc[8][2];
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    m[i] = -INFINITY;
    l[i] = 0.f;
    acc[i][0] = acc[i][1] = 0ull;
  }

  for (int t = grp; t < ntiles; t += G) {
    copy_wait<0>();                                          // K of this tile
    group_sync();
    f32x2 s2[8][4];
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) s2[i][j] = 0ull;
#pragma unroll 4
    for (int c = 0; c < kDim; c += 4) {
      ulonglong2 kk[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) kk[j] = *reinterpret_cast<const ulonglong2*>(kg + (tx + 16 * j) * kLd + c);
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const ulonglong2 qq = *reinterpret_cast<const ulonglong2*>(qr + i * kLd + c);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          fma2(s2[i][j], qq.x, kk[j].x);
          fma2(s2[i][j], qq.y, kk[j].y);
        }
      }
    }
    group_sync();                                            // the group is done with K
    load_tile(kg, v, t);                                     // V, under the softmax

    const bool ragged = (t + 1) * kKeys > cnt;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      float s[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float2 e = unpack2(s2[i][j]);
        s[j] = (e.x + e.y) * scale;
        if (ragged && t * kKeys + tx + 16 * j >= cnt) s[j] = -INFINITY;
      }
      float mx = fmaxf(fmaxf(s[0], s[1]), fmaxf(s[2], s[3]));
#pragma unroll
      for (int w = 1; w < 16; w <<= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, w));
      const float mn = fmaxf(m[i], mx);                      // finite: every tile holds at least one key
      const float alpha = expf(m[i] - mn);                   // exp(-inf) = 0 on the first tile
      m[i] = mn;
      float sum = 0.f;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float p = expf(s[j] - mn);
        sum += p;
        pw[(ty * 8 + i) * kLd + tx + 16 * j] = p;
      }
      l[i] = fmaf(l[i], alpha, sum);
      const f32x2 a2 = pack2(alpha, alpha);
      acc[i][0] = mul2(acc[i][0], a2);
      acc[i][1] = mul2(acc[i][1], a2);
    }
    copy_wait<0>();                                          // V of this tile
    group_sync();                                            // (also orders the warp's own probabilities)
#pragma unroll 4
    for (int c = 0; c < kKeys; c += 4) {
      ulonglong2 vv[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) vv[j] = *reinterpret_cast<const ulonglong2*>(kg + (c + j) * kLd + 4 * tx);
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const float4 pp = *reinterpret_cast<const float4*>(pw + (ty * 8 + i) * kLd + c);
        const f32x2 p0 = pack2(pp.x, pp.x), p1 = pack2(pp.y, pp.y), p2 = pack2(pp.z, pp.z), p3 = pack2(pp.w, pp.w);
        fma2(acc[i][0], p0, vv[0].x);
        fma2(acc[i][1], p0, vv[0].y);
        fma2(acc[i][0], p1, vv[1].x);
        fma2(acc[i][1], p1, vv[1].y);
        fma2(acc[i][0], p2, vv[2].x);
        fma2(acc[i][1], p2, vv[2].y);
        fma2(acc[i][0], p3, vv[3].x);
        fma2(acc[i][1], p3, vv[3].y);
      }
    }
    group_sync();                                            // the group is done with V (and the warp with its P)
    if (t + G < ntiles) load_tile(kg, k, t + G);
  }

#pragma unroll
  for (int i = 0; i < 8; ++i) {
#pragma unroll
    for (int w = 1; w < 16; w <<= 1) l[i] += __shfl_xor_sync(0xffffffffu, l[i], w);
  }
  // Merge the groups through the warps' own buffers: output channels 0..63 of a row, then its maximum and sum.
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    float* dst = pw + (ty * 8 + i) * kLd;
    ulonglong2 x;
    x.x = acc[i][0];
    x.y = acc[i][1];
    *reinterpret_cast<ulonglong2*>(dst + 4 * tx) = x;
    if (tx == 0) {
      dst[64] = m[i];
      dst[65] = l[i];
    }
  }
  __syncthreads();
  constexpr int kOwnRows = kRowsWarp / G;                    // rows of row warp rw that this warp writes out
#pragma unroll
  for (int j = 0; j < kOwnRows / 2; ++j) {
    const int r = grp * kOwnRows + 2 * j + ty, row = row0 + rw * kRowsWarp + r;
    if (row < nq) {
      float M = -INFINITY;
#pragma unroll
      for (int g = 0; g < G; ++g) M = fmaxf(M, ps[((g * R + rw) * kRowsWarp + r) * kLd + 64]);
      float L = 0.f;
      float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int g = 0; g < G; ++g) {
        const float* src = ps + ((g * R + rw) * kRowsWarp + r) * kLd;
        const float f = expf(src[64] - M);                   // a group without a tile: exp(-inf) = 0
        const float4 y = *reinterpret_cast<const float4*>(src + 4 * tx);
        L = fmaf(src[65], f, L);
        x.x = fmaf(y.x, f, x.x);
        x.y = fmaf(y.y, f, x.y);
        x.z = fmaf(y.z, f, x.z);
        x.w = fmaf(y.w, f, x.w);
      }
      const float inv = 1.f / L;
      const int tok = key_token(prefix_rows ? row : P + row);
      *reinterpret_cast<float4*>(o + base + (size_t)tok * kDim + 4 * tx) = make_float4(x.x * inv, x.y * inv, x.z * inv, x.w * inv);
    }
  }
  if (overlap) griddep_wait();
}

template <int R, int G>
cudaError_t launch(const AttnArgs& a, bool prefix_rows, bool overlap, cudaStream_t st) {
  static OncePerDevice opt_in;
  const cudaError_t e = opt_in.run([&] {
    return cudaFuncSetAttribute(attn_f32_kernel<R, G>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_bytes<R, G>());
  });
  if (e != cudaSuccess) return e;
  const int wh = a.wh < a.Hg ? a.wh : a.Hg, ww = a.ww < a.Wg ? a.ww : a.Wg;
  const int nwx = ceil_div(a.Wg, ww), nwin = nwx * ceil_div(a.Hg, wh);
  const dim3 grid = prefix_rows ? dim3(ceil_div(a.P, R * kRowsWarp), 1, a.BH) : dim3(ceil_div(wh * ww, R * kRowsWarp), nwin, a.BH);
  return launch_programmatic(attn_f32_kernel<R, G>, grid, 32 * R * G, smem_bytes<R, G>(), st, (const float*)a.q, (const float*)a.k,
                             (const float*)a.v, (float*)a.o, a.Hg, a.Wg, a.P, wh, ww, nwx, prefix_rows, overlap, a.scale);
}

}  // namespace

bool attn_f32_supported(const AttnArgs& a) { return a.dtype == JV_F32 && a.D == kDim && !a.strided; }

// The P prefix queries go first, with the keys of a row tile split over four groups (their chain is the
// longest: all N keys); the windows' launch overlaps them, as neither reads what the other writes.
// 32 rows x 2 groups per CTA, unless that leaves the chip nearly empty: then 16 rows x 4 groups, which halves a CTA's
// chain.  Measured, 32 x 2 against 16 x 4: 48 CTAs of 32 rows 16 / 10 us, 156 CTAs 39 / 34 us, 258 CTAs 98 / 110 us, 384 CTAs
// 103 / 115 us; windows of one or two key tiles have no work for four groups (432 CTAs, 8 x 8 windows: 18 / 33 us).
cudaError_t launch_attn_f32(const AttnArgs& a, cudaStream_t st) {
  const int wh = a.wh < a.Hg ? a.wh : a.Hg, ww = a.ww < a.Wg ? a.ww : a.Wg;
  const bool prefix = a.P > 0;
  if (prefix) {
    const cudaError_t e = launch<1, 4>(a, true, false, st);
    if (e != cudaSuccess) return e;
  }
  const int64_t ctas = (int64_t)ceil_div(a.Wg, ww) * ceil_div(a.Hg, wh) * a.BH * ceil_div(wh * ww, 2 * kRowsWarp);
  if (4 * ctas <= 5 * device_sm_count() && wh * ww + a.P > 2 * kKeys) return launch<1, 4>(a, false, prefix, st);
  return launch<2, 2>(a, false, prefix, st);
}

}  // namespace jv
