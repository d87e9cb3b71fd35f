// The prefix queries of window attention (Sec. 3.2.2): the P prefix tokens of a (batch, head) attend all its P + N tokens.
// bf16 tensors, head_dim 64.
//
// A handful of query rows against thousands of keys: what bounds it is reading K and V once, so the keys are spread over
// the chip and everything is laid out for loads in flight.  mma.sync m16n8k16 with a group of up to 16 query rows as the M
// dimension; a cluster of 1, 2, 4 or 8 CTAs serves one (batch, head) and
// group, its warps take 16-key tiles round-robin.  K and V
// go from global memory straight into the MMA's B fragments, 128 bits per load, the next tile's on their way while this
// one is worked on; the layouts are free to be what such loads give:
//   scores   lane (g, t) holds channels 16 t .. 16 t + 15 of key g of an 8-key group; channels may meet in any order, so
//            Q's fragments take the same one
//   P V      lane (g, t) holds channels 8 g .. 8 g + 7 of keys 2 t, 2 t + 1, 2 t + 8, 2 t + 9; product j yields channel
//            8 n + j in column n
// The partial results (maximum, sum, weighted V per row) are merged in two steps: the warps of a CTA through its shared
// memory, the CTAs of the cluster through distributed shared memory.  No scratch in global memory, no atomics: bit-reproducible.
//
// Measured, 8 x 16 heads, 5 prefix and 64 x 64 grid tokens: 28.8 us = 4.7 TB/s (what a plain read of this size reaches) against
// 41.5 with the tiles staged through shared memory and two CTAs per head; 6 heads, 37 x 37 tokens: 6 us against 15.  Two tiles
// ahead instead of one costs a CTA per SM and 46.9 us; sixteen warps per CTA are no faster.
#include <cooperative_groups.h>

#include "common.cuh"

namespace jv {
namespace {

constexpr int kRows = 16;                             // query rows per group
constexpr int kD = 64;
constexpr int kWarps = 8;
constexpr int kKeys = 16;                             // keys per warp and step
constexpr int kLd = 2 + kD;                           // a row's partial: maximum, sum, 64 weighted channels

__device__ __forceinline__ void mma16816(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
               : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
  __nv_bfloat162 t = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&t);
}

struct Tile {
  uint4 k[2][2], v[4];                                // keys g, g + 8: channels 16 t ..; keys 2 t, 2 t + 1, 2 t + 8, 2 t + 9: channels 8 g ..
};

__global__ void __launch_bounds__(kWarps * 32, 2)
attn_prefix_rows_kernel(const __nv_bfloat16* __restrict__ q, const __nv_bfloat16* __restrict__ k,
                        const __nv_bfloat16* __restrict__ v, __nv_bfloat16* __restrict__ o, const int* status, int N, int P,
                        float scale_log2) {
  namespace cg = cooperative_groups;
  __shared__ float part[kWarps + 1][kRows][kLd];      // one partial per warp, then the block's own
  griddep_wait();
  griddep_launch_dependents();                        // the windows' launch overlaps this one
  const bool gave_up = *reinterpret_cast<const volatile int*>(status) != 0;   // an earlier kernel gave up: o stays as it is
  cg::cluster_group cluster = cg::this_cluster();
  const int nsplit = cluster.num_blocks(), split = cluster.block_rank();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int r0 = blockIdx.y * kRows, nr = min(kRows, P - r0);
  const size_t base = (size_t)(blockIdx.x / nsplit) * N * kD;
  const uint4 zero = make_uint4(0u, 0u, 0u, 0u);
  // Eight channels of a token.  A coherent load: beside the windows this launch may start while the one ahead of it still
  // writes q, k and v, and a non-coherent one promises that nobody does for as long as the kernel runs.
  auto row16 = [&](const __nv_bfloat16* src, int row, int ch, bool in) -> uint4 {
    return in ? __ldcg(reinterpret_cast<const uint4*>(src + base + (size_t)row * kD + ch)) : zero;
  };
  auto load = [&](Tile& x, int t0) {
#pragma unroll
    for (int n = 0; n < 2; ++n) {
      const int key = t0 + 8 * n + g;
      x.k[n][0] = row16(k, key, 16 * t, key < N);
      x.k[n][1] = row16(k, key, 16 * t + 8, key < N);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int key = t0 + 2 * t + (i & 1) + 8 * (i >> 1);
      x.v[i] = row16(v, key, 8 * g, key < N);
    }
  };
  const int step = nsplit * kWarps * kKeys;
  int t0 = (split * kWarps + warp) * kKeys;
  Tile cur;
  load(cur, t0);                                      // (all zeros past the last key)
  uint32_t qa[4][4];                                  // A fragments of Q, [k step][row g | row g + 8 | ...]: zeros past P
  {
    const uint4 a0 = row16(q, r0 + g, 16 * t, g < nr), a1 = row16(q, r0 + g, 16 * t + 8, g < nr);
    const uint4 b0 = row16(q, r0 + g + 8, 16 * t, g + 8 < nr), b1 = row16(q, r0 + g + 8, 16 * t + 8, g + 8 < nr);
    const uint32_t a[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w}, b[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
#pragma unroll
    for (int s = 0; s < 4; ++s) {                     // step s: channels 16 t + 4 s .. + 3
      qa[s][0] = a[2 * s]; qa[s][1] = b[2 * s]; qa[s][2] = a[2 * s + 1]; qa[s][3] = b[2 * s + 1];
    }
  }
  float m[2] = {-INFINITY, -INFINITY}, l[2] = {0.f, 0.f};            // rows g and g + 8
  float acc[8][4];
#pragma unroll
  for (int j = 0; j < 8; ++j)
#pragma unroll
    for (int c = 0; c < 4; ++c) acc[j][c] = 0.f;

  for (; t0 < N; t0 += step) {
    Tile nxt;
    load(nxt, t0 + step);
    float sc[2][4];
#pragma unroll
    for (int n = 0; n < 2; ++n) {
#pragma unroll
      for (int c = 0; c < 4; ++c) sc[n][c] = 0.f;
      const uint32_t b[8] = {cur.k[n][0].x, cur.k[n][0].y, cur.k[n][0].z, cur.k[n][0].w, cur.k[n][1].x, cur.k[n][1].y, cur.k[n][1].z, cur.k[n][1].w};
#pragma unroll
      for (int s = 0; s < 4; ++s) mma16816(sc[n], qa[s], b[2 * s], b[2 * s + 1]);
    }
    // online softmax of rows g (c0, c1) and g + 8 (c2, c3); key of element c: t0 + 8 n + 2 t + (c & 1)
    float mx[2] = {-INFINITY, -INFINITY};
#pragma unroll
    for (int n = 0; n < 2; ++n)
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        sc[n][c] = t0 + 8 * n + 2 * t + (c & 1) < N ? sc[n][c] * scale_log2 : -INFINITY;
        mx[c >> 1] = fmaxf(mx[c >> 1], sc[n][c]);
      }
    float alpha[2], ref[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      mx[h] = fmaxf(mx[h], __shfl_xor_sync(0xffffffffu, mx[h], 1));
      mx[h] = fmaxf(mx[h], __shfl_xor_sync(0xffffffffu, mx[h], 2));
      const float m_new = fmaxf(m[h], mx[h]);
      ref[h] = m_new == -INFINITY ? 0.f : m_new;                     // all scores of this warp so far are -inf: weight 0, not NaN
      alpha[h] = exp2f(m[h] - ref[h]);
      m[h] = m_new;
      l[h] *= alpha[h];                                              // (this lane's share of the sum)
    }
    uint32_t pa[4];                                                  // A fragment of P
#pragma unroll
    for (int n = 0; n < 2; ++n) {
      const float p0 = exp2f(sc[n][0] - ref[0]), p1 = exp2f(sc[n][1] - ref[0]);
      const float p2 = exp2f(sc[n][2] - ref[1]), p3 = exp2f(sc[n][3] - ref[1]);
      l[0] += p0 + p1;
      l[1] += p2 + p3;
      pa[2 * n] = pack_bf16x2(p0, p1);                               // row g
      pa[2 * n + 1] = pack_bf16x2(p2, p3);                           // row g + 8
    }
    const uint32_t w[4][4] = {{cur.v[0].x, cur.v[0].y, cur.v[0].z, cur.v[0].w}, {cur.v[1].x, cur.v[1].y, cur.v[1].z, cur.v[1].w},
                              {cur.v[2].x, cur.v[2].y, cur.v[2].z, cur.v[2].w}, {cur.v[3].x, cur.v[3].y, cur.v[3].z, cur.v[3].w}};
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      acc[j][0] *= alpha[0]; acc[j][1] *= alpha[0];
      acc[j][2] *= alpha[1]; acc[j][3] *= alpha[1];
      const uint32_t sel = (j & 1) ? 0x7632u : 0x5410u;              // channel 8 g + j of two keys side by side
      mma16816(acc[j], pa, __byte_perm(w[0][j >> 1], w[1][j >> 1], sel), __byte_perm(w[2][j >> 1], w[3][j >> 1], sel));
    }
    cur = nxt;
  }
  // merge, step 1: the warps of this block
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    l[h] += __shfl_xor_sync(0xffffffffu, l[h], 1);
    l[h] += __shfl_xor_sync(0xffffffffu, l[h], 2);
    float* dst = part[warp][g + 8 * h];
    if (t == 0) { dst[0] = m[h]; dst[1] = l[h]; }
#pragma unroll
    for (int j = 0; j < 8; ++j) {                                    // columns 2 t, 2 t + 1 of product j: channels 16 t + j, 16 t + 8 + j
      dst[2 + 16 * t + j] = acc[j][2 * h];
      dst[2 + 16 * t + 8 + j] = acc[j][2 * h + 1];
    }
  }
  __syncthreads();
  // n partials combined into (M, L, two channels per lane)
  auto combine = [&](int n, auto&& src_of, float& M, float& L, float& x0, float& x1) {
    M = -INFINITY; L = 0.f; x0 = 0.f; x1 = 0.f;
    for (int i = 0; i < n; ++i) M = fmaxf(M, src_of(i)[0]);
    for (int i = 0; i < n; ++i) {
      const float* src = src_of(i);
      const float f = src[0] == -INFINITY ? 0.f : exp2f(src[0] - M);   // a source that saw no key, or none of weight
      L = fmaf(src[1], f, L);
      x0 = fmaf(src[2 + lane], f, x0);
      x1 = fmaf(src[2 + 32 + lane], f, x1);
    }
  };
  for (int r = warp; r < nr; r += kWarps) {
    float M, L, x0, x1;
    combine(kWarps, [&](int i) { return part[i][r]; }, M, L, x0, x1);
    float* dst = part[kWarps][r];
    if (lane == 0) { dst[0] = M; dst[1] = L; }
    dst[2 + lane] = x0;
    dst[2 + 32 + lane] = x1;
  }
  // step 2: the blocks of the cluster, rows dealt out over its blocks and warps
  cluster.sync();
  for (int r = split * kWarps + warp; r < nr; r += nsplit * kWarps) {
    float M, L, x0, x1;
    combine(nsplit, [&](int i) { return cluster.map_shared_rank(&part[kWarps][r][0], i); }, M, L, x0, x1);
    const float inv = 1.f / L;
    __nv_bfloat16* dst = o + base + (size_t)(r0 + r) * kD;
    if (!gave_up) {
      dst[lane] = __float2bfloat16_rn(x0 * inv);
      dst[32 + lane] = __float2bfloat16_rn(x1 * inv);
    }
  }
  cluster.sync();                                     // no block leaves while its shared memory may still be read
}

}  // namespace

// To be enqueued right ahead of the windows' launch, which may overlap it (neither reads what the other writes) and ends
// only after it: this one is short and, on small problems, leaves most SMs free.  Behind the windows it took 2 us of its own
// even there (6 heads, 37 x 37 tokens), and a persistent kernel of the windows leaves it no SM until it ends.
// ctas: how many blocks it should have at most (it has at least one per (batch, head) and group).
//
// Beside the windows, on the SMs that their launch leaves free, if there is a block for every head and none has more than 24 steps to
// walk; else on the whole chip ahead of them.  Measured, beside / ahead: 24 heads, 48 x 48 tokens, 40 SMs free, 18 steps: 15.5 / 20.6 us
// for the call; 16 heads, 64 x 64, 20 SMs free, 33 steps: 23.1 / 20.6.
// Ahead, the launch is a plain one: dropped in while the launch before it drains, its blocks fill the first SMs two to one
// and leave the last without.  Programmatically / plainly: 8 x 16 heads, 64 x 64 tokens 97.5 / 90.9 us for the call, 16 heads, 128 x 128
// tokens 64.8 / 58.5, 24 heads, 40 x 60 22.0 / 22.9; beside, 6 heads, 37 x 37: 11.9 / 14.1.
cudaError_t launch_attn_prefix(const AttnArgs& a, int free_sms, const int* status, cudaStream_t st) {
  if (a.dtype != JV_BF16 || a.D != kD || a.strided) return cudaErrorNotSupported;   // (the callers are the bf16 tensor-core paths)
  const int N = a.P + a.Hg * a.Wg, groups = ceil_div(a.P, kRows);
  // splits of the keys over at most `ctas` blocks: at least one 16-key step per warp
  auto split_for = [&](int64_t ctas) {
    int split = 1;
    while (split < 8 && 2ll * split * a.BH * groups <= ctas && split * kWarps * kKeys < N) split *= 2;
    return split;
  };
  int split = split_for(free_sms);
  const bool beside = (int64_t)a.BH * groups <= free_sms && ceil_div(N, split * kWarps * kKeys) <= 24;
  if (!beside) split = split_for(2 * device_sm_count());
  const dim3 grid(a.BH * split, groups);
  return launch_cluster(beside, attn_prefix_rows_kernel, split, grid, kWarps * 32, 0, st,
                        (const __nv_bfloat16*)a.q, (const __nv_bfloat16*)a.k, (const __nv_bfloat16*)a.v, (__nv_bfloat16*)a.o, status, N, a.P,
                        a.scale * 1.4426950408889634f);
}

}  // namespace jv
