// Linear attention (Sec. 3.2.1, Eq. 2 reordered) at head_dim 128 on the tensor cores: bf16 tensors, no convolution.
//
//   lin128_state_kernel   per (head, token chunk): KV = relu(K)^T V, z = relu(K)^T 1 (mma.sync m16n8k16, TMA ring).
//                         The chunks of a head are one thread-block cluster: their partial states are summed in
//                         chunk order through distributed shared memory (no atomics: bit-reproducible), and the
//                         finished state is written once, as the apply pass wants it: KV as a sum of kSplit bf16
//                         matrices, each already in the 128-byte-swizzled layout of its MMA operand, z in fp32.
//   lin128_apply_kernel   o = relu(q) KV / (relu(q) . z + eps) per 128-token tile: one bulk copy of the state, ReLU in place in
//                         shared memory, tcgen05.mma with the accumulator in tensor memory, TMA stores.
//
// What bounds it: HBM (K, V, Q read once, O written once: 1 KB per token and head).  At this head_dim the
// summed state is 66 KB per head: summing chunk partials in every apply CTA, as at head_dim 64, would read more than Q,
// hence the cluster reduction.  KV as three bf16 terms keeps the 24 bits of the fp32 state, so the product
// is as exact as the fp32 kernels' that served these calls before.
// Measured, 2 x 8 heads, 64 x 64 tokens: MEASURED
#include <cooperative_groups.h>

#include "lin_common.cuh"

namespace jv {
namespace {

using namespace tc;
using lin::griddep_launch_dependents;
using lin::griddep_wait;
using lin::relu_bf16x2;
using lin::bf16x2_to_f2;
using lin::tile_off;

constexpr int kC = 128;                               // channels per head
constexpr int kSplit = 3;                             // bf16 terms of KV
constexpr int kKvHalf = kC * 64 * 2;                  // one 64-column half of one term: 128 rows of 128 bytes
constexpr int kKvBytes = kSplit * 2 * kKvHalf;        // [term][column half][row a][64 columns]
constexpr size_t kStateBytes = (size_t)kKvBytes + kC * sizeof(float);   // per (batch, head): KV, then z

// ---- state pass -------------------------------------------------------------------
constexpr int kTok1 = 64;                             // tokens per tile
constexpr int kHalf1 = kTok1 * 128;                   // 64 tokens x 64 channels: 8 KB
constexpr int kStage1 = 4 * kHalf1;                   // K (two halves), V (two halves)
constexpr int kStages1 = 3;
constexpr int kMmaWarps = 8;
constexpr int kThreads1 = (kMmaWarps + 1) * 32;
constexpr int kLdRed = kC + 4;                        // padded row of the partial state in shared memory (over the ring)
constexpr int kMaxCluster = 8;
struct __align__(8) Bars1 {
  uint64_t full[kStages1], empty[kStages1];
  volatile uint32_t abort_flag;
  float z[kC];
};
constexpr size_t kSmem1 = (size_t)kStages1 * kStage1 + sizeof(Bars1) + 1024;
static_assert((size_t)kC * kLdRed * sizeof(float) <= (size_t)kStages1 * kStage1, "the partial state fits over the ring");

__device__ __forceinline__ void ldmatrix_x4_trans(uint32_t (&r)[4], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
__device__ __forceinline__ void mma_bf16(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
               : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

__global__ void __launch_bounds__(kThreads1, 2)
lin128_state_kernel(const __grid_constant__ CUtensorMap mapK, const __grid_constant__ CUtensorMap mapV,
                    unsigned char* __restrict__ state, int* status, int N, int chunk_tokens) {
  namespace cg = cooperative_groups;
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem_al = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  const uint32_t smem = smem_u32(smem_al);
  Bars1* bars = reinterpret_cast<Bars1*>(smem_al + (size_t)kStages1 * kStage1);
  cg::cluster_group cluster = cg::this_cluster();
  const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
  const int bh = blockIdx.y, chunk = blockIdx.x, nchunk = gridDim.x;   // the cluster is the whole grid row
  const int t_begin = min(N, chunk * chunk_tokens), t_end = min(N, t_begin + chunk_tokens);
  const int ntiles = (t_end - t_begin + kTok1 - 1) / kTok1;            // 0 for a chunk past the end

  griddep_launch_dependents();
  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages1; ++s) {
      mbar_init(&bars->full[s], 1);
      mbar_init(&bars->empty[s], kMmaWarps);
    }
    // an earlier kernel gave up: no copies, no waits (but this CTA still takes part in the cluster's barriers)
    bars->abort_flag = *reinterpret_cast<volatile int*>(status) != 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  __syncthreads();
  bool ok = bars->abort_flag == 0;

  // warp w of the eight: rows 32 (w / 2) .. + 31 of KV, columns 64 (w % 2) .. + 63
  const int rg = warp >> 1, ch = warp & 1;
  float acc[2][8][4], accz[2][4];
#pragma unroll
  for (int m = 0; m < 2; ++m) {
#pragma unroll
    for (int j = 0; j < 8; ++j)
#pragma unroll
      for (int i = 0; i < 4; ++i) acc[m][j][i] = 0.f;
#pragma unroll
    for (int i = 0; i < 4; ++i) accz[m][i] = 0.f;
  }
  if (warp == kMmaWarps) {
    // ================= TMA producer =================
    int issued = 0;
    for (int it = 0; it < ntiles && ok; ++it) {
      const int s = it % kStages1;
      if (it >= kStages1) ok = warp_wait(&bars->empty[s], ((it / kStages1) - 1) & 1, &bars->abort_flag, status);
      if (!ok) break;
      if (elect_one()) {
        mbar_expect_tx(&bars->full[s], kStage1);
        const int tok = t_begin + it * kTok1;               // rows past N arrive as zeros
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          tma_load_3d(smem + s * kStage1 + h * kHalf1, &mapK, &bars->full[s], 64 * h, tok, bh);
          tma_load_3d(smem + s * kStage1 + (2 + h) * kHalf1, &mapV, &bars->full[s], 64 * h, tok, bh);
        }
      }
      __syncwarp();
      ++issued;
    }
    if (!ok && lane == 0) {   // let the copies in flight land before the CTA leaves
      const unsigned long long t0 = globaltimer();
      for (int g = max(0, issued - kStages1); g < issued; ++g)
        while (!mbar_try(&bars->full[g % kStages1], (g / kStages1) & 1) && globaltimer() - t0 < kWaitLimitNs) {}
    }
    __syncwarp();
  } else {
    const uint32_t ones = (lane < 4) ? 0x3F803F80u : 0u;    // B fragment of a ones column
    for (int it = 0; it < ntiles && ok; ++it) {
      const int s = it % kStages1;
      ok = warp_wait(&bars->full[s], (it / kStages1) & 1, &bars->abort_flag, status);
      if (!ok) break;
      const uint32_t ks = smem + s * kStage1 + (rg >> 1) * kHalf1, vsm = smem + s * kStage1 + (2 + ch) * kHalf1;
#pragma unroll
      for (int kk = 0; kk < kTok1 / 16; ++kk) {
        uint32_t a[2][4];
        const int ta = kk * 16 + (lane & 7) + ((lane >> 4) & 1) * 8;
#pragma unroll
        for (int m = 0; m < 2; ++m) {                       // A = relu(K)^T; K is stored [token][a] -> .trans
          ldmatrix_x4_trans(a[m], ks + tile_off(ta, 4 * (rg & 1) + 2 * m + ((lane >> 3) & 1)));
#pragma unroll
          for (int i = 0; i < 4; ++i) a[m][i] = relu_bf16x2(a[m][i]);
        }
        const int tb = kk * 16 + (lane & 7) + ((lane >> 3) & 1) * 8;
#pragma unroll
        for (int jp = 0; jp < 4; ++jp) {
          uint32_t b[4];                                    // V stored [token][e] -> .trans; two n-tiles per load
          ldmatrix_x4_trans(b, vsm + tile_off(tb, 2 * jp + (lane >> 4)));
#pragma unroll
          for (int m = 0; m < 2; ++m) {
            mma_bf16(acc[m][2 * jp], a[m], b[0], b[1]);
            mma_bf16(acc[m][2 * jp + 1], a[m], b[2], b[3]);
          }
        }
        if (ch == 0) {
#pragma unroll
          for (int m = 0; m < 2; ++m) mma_bf16(accz[m], a[m], ones, ones);
        }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&bars->empty[s]);
    }
  }
  // every copy has been waited for by the MMA warps (or landed above): the ring becomes the partial state
  __syncthreads();
  float* red = reinterpret_cast<float*>(smem_al);
  const int g = lane >> 2, tq = lane & 3;
  if (warp < kMmaWarps) {
#pragma unroll
    for (int m = 0; m < 2; ++m) {
      const int a0 = 32 * rg + 16 * m + g;
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        *reinterpret_cast<float2*>(red + a0 * kLdRed + 64 * ch + 8 * j + 2 * tq) = make_float2(acc[m][j][0], acc[m][j][1]);
        *reinterpret_cast<float2*>(red + (a0 + 8) * kLdRed + 64 * ch + 8 * j + 2 * tq) = make_float2(acc[m][j][2], acc[m][j][3]);
      }
      if (ch == 0 && tq == 0) {
        bars->z[a0] = accz[m][0];
        bars->z[a0 + 8] = accz[m][2];
      }
    }
  }
  cluster.sync();
  // this CTA finishes rows chunk * rows .. + rows - 1 of the head's state, eight columns per thread
  const int rows = kC / nchunk, row0 = chunk * rows;
  unsigned char* st = state + (size_t)bh * kStateBytes;
  for (int i = threadIdx.x; i < rows * (kC / 8); i += kThreads1) {
    const int row = row0 + i / (kC / 8), c8 = i % (kC / 8);
    float x[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) x[e] = 0.f;
#pragma unroll
    for (int c = 0; c < kMaxCluster; ++c) {
      if (c < nchunk) {
        const float* src = cluster.map_shared_rank(red, c) + row * kLdRed + 8 * c8;
        const float4 lo = *reinterpret_cast<const float4*>(src), hi = *reinterpret_cast<const float4*>(src + 4);
        x[0] += lo.x; x[1] += lo.y; x[2] += lo.z; x[3] += lo.w;
        x[4] += hi.x; x[5] += hi.y; x[6] += hi.z; x[7] += hi.w;
      }
    }
#pragma unroll
    for (int s = 0; s < kSplit; ++s) {                      // the bf16 nearest to what the terms before it left over
      uint32_t w[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        w[e] = pack_bf16(x[2 * e], x[2 * e + 1]);
        const float2 f = bf16x2_to_f2(w[e]);
        x[2 * e] -= f.x;
        x[2 * e + 1] -= f.y;
      }
      *reinterpret_cast<uint4*>(st + (size_t)(2 * s + (c8 >> 3)) * kKvHalf + tile_off(row, c8 & 7)) = make_uint4(w[0], w[1], w[2], w[3]);
    }
  }
  for (int i = threadIdx.x; i < rows; i += kThreads1) {
    float z = 0.f;
    for (int c = 0; c < nchunk; ++c) z += cluster.map_shared_rank(bars->z, c)[row0 + i];
    reinterpret_cast<float*>(st + kKvBytes)[row0 + i] = z;
  }
  cluster.sync();                                           // no CTA leaves while its partial may still be read
}

// ---- apply pass ---------------------------------------------------------------------
constexpr int kTok2 = 128;                            // tokens per tile
constexpr int kHalf2 = kTok2 * 128;                   // 128 tokens x 64 channels: 16 KB
constexpr int kTile2 = 2 * kHalf2;
constexpr int kSlots = 3;                             // Q tiles; a slot becomes its tile's output staging
constexpr int kThreads2 = 288;                        // 4 rectifier warps, 1 producer / issuer warp, 4 epilogue warps
constexpr uint32_t kTmemCols = 256;                   // two 128-column fp32 accumulators
struct __align__(8) Bars2 {
  uint64_t q_full[kSlots], q_free[kSlots];            // TMA landed / the four store groups have read the slot
  uint64_t relu_done[kSlots];                         // 128 arrivals: the tile is rectified, its denominators stored
  uint64_t d_full[2], d_empty[2];                     // accumulator complete / read by the epilogue (128 arrivals)
  uint64_t kv_full;                                   // the state has landed
  uint32_t tmem_base;
  volatile uint32_t abort_flag;
};
constexpr size_t kOffQ = kKvBytes, kOffZ2 = kOffQ + (size_t)kSlots * kTile2, kOffDen = kOffZ2 + kC * sizeof(float);
constexpr size_t kOffBars2 = kOffDen + (size_t)kSlots * kTok2 * sizeof(float);
constexpr size_t kSmem2 = kOffBars2 + sizeof(Bars2) + 1024;
static_assert(kSmem2 <= 232448, "shared memory of one CTA");
constexpr uint32_t kIdesc = idesc(128, 64, 1);        // D fp32, A and B bf16, B MN-major, M = 128, N = 64

__global__ void __launch_bounds__(kThreads2, 1)
lin128_apply_kernel(const __grid_constant__ CUtensorMap mapQ, const __grid_constant__ CUtensorMap mapO,
                    const unsigned char* __restrict__ state, int* status, int N, int span_tokens, float eps) {
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem_al = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  const uint32_t smem = smem_u32(smem_al);
  float* z_sm = reinterpret_cast<float*>(smem_al + kOffZ2);
  float* den_sm = reinterpret_cast<float*>(smem_al + kOffDen);        // [kSlots][128]
  Bars2* bars = reinterpret_cast<Bars2*>(smem_al + kOffBars2);
  const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
  const int bh = blockIdx.y;
  const int t_begin = blockIdx.x * span_tokens, t_end = min(N, t_begin + span_tokens);
  const int ntiles = (t_end - t_begin + kTok2 - 1) / kTok2;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kSlots; ++s) {
      mbar_init(&bars->q_full[s], 1);
      mbar_init(&bars->q_free[s], 4);
      mbar_init(&bars->relu_done[s], 128);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&bars->d_full[b], 1);
      mbar_init(&bars->d_empty[b], 128);
    }
    mbar_init(&bars->kv_full, 1);
    bars->abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 0) {
    __syncwarp();
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&bars->tmem_base)),
                 "r"(kTmemCols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = __shfl_sync(0xffffffffu, bars->tmem_base, 0);
  bool ok = true;

  if (warp == 4) {
    // ================= TMA producer and MMA issuer =================
    int issued = 0;
    bool kv_issued = false;
    auto load_tile = [&](int it) {
      if (elect_one()) {
        const int s = it % kSlots;
        mbar_expect_tx(&bars->q_full[s], kTile2);
        tma_load_3d(smem + (uint32_t)kOffQ + s * kTile2, &mapQ, &bars->q_full[s], 0, t_begin + it * kTok2, bh);
        tma_load_3d(smem + (uint32_t)kOffQ + s * kTile2 + kHalf2, &mapQ, &bars->q_full[s], 64, t_begin + it * kTok2, bh);
      }
      __syncwarp();
      ++issued;
    };
    for (int it = 0; it < kSlots && it < ntiles; ++it) load_tile(it);   // Q does not depend on the state pass
    griddep_wait();                                    // the state pass is complete
    if (*reinterpret_cast<volatile int*>(status) != 0) {
      bars->abort_flag = 1;                            // an earlier kernel gave up: every role falls through
      ok = false;
    } else {
      kv_issued = true;
      if (elect_one()) {
        mbar_expect_tx(&bars->kv_full, kKvBytes + kC * 4);
        asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                     ::"r"(smem), "l"(state + (size_t)bh * kStateBytes), "r"(kKvBytes), "r"(smem_u32(&bars->kv_full)) : "memory");
        asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                     ::"r"(smem_u32(z_sm)), "l"(state + (size_t)bh * kStateBytes + kKvBytes), "r"(kC * 4),
                       "r"(smem_u32(&bars->kv_full)) : "memory");
      }
      __syncwarp();
      ok = warp_wait(&bars->kv_full, 0, &bars->abort_flag, status);
    }
    for (int it = 0; it < ntiles && ok; ++it) {
      const int s = it % kSlots, b = it & 1;
      ok = warp_wait(&bars->relu_done[s], (it / kSlots) & 1, &bars->abort_flag, status);
      if (ok && it >= 2) ok = warp_wait(&bars->d_empty[b], ((it >> 1) - 1) & 1, &bars->abort_flag, status);
      if (!ok) break;
      tc_fence_after();
      if (elect_one()) {
        const uint32_t qa = smem + (uint32_t)kOffQ + s * kTile2;
#pragma unroll 1
        for (int h = 0; h < 2; ++h)                    // 64-column halves of the accumulator
#pragma unroll 1
          for (int x = 0; x < kSplit; ++x) {
            const uint64_t da = smem_desc(qa), db = smem_desc(smem + (2 * x + h) * kKvHalf);
#pragma unroll
            for (int ks = 0; ks < kC / 16; ++ks)
              mma_ss_1(tmem + b * kC + 64 * h, desc_advance(da, (ks >> 2) * kHalf2 + (ks & 3) * 32), desc_advance(db, ks * 2048),
                       kIdesc, (x > 0 || ks > 0) ? 1u : 0u);
          }
      }
      __syncwarp();
      tc_commit(&bars->d_full[b]);
      const int nx = it + kSlots - 1;                  // into the slot of tile it - 1, once its stores have read it
      if (it > 0 && nx < ntiles) {
        ok = warp_wait(&bars->q_free[nx % kSlots], ((it - 1) / kSlots) & 1, &bars->abort_flag, status);
        if (!ok) break;
        load_tile(nx);
      }
    }
    if (!ok && lane == 0) {                            // let the copies in flight land before the CTA leaves
      const unsigned long long t0 = globaltimer();
      for (int g = max(0, issued - kSlots); g < issued; ++g)
        while (!mbar_try(&bars->q_full[g % kSlots], (g / kSlots) & 1) && globaltimer() - t0 < kWaitLimitNs) {}
      while (kv_issued && !mbar_try(&bars->kv_full, 0) && globaltimer() - t0 < kWaitLimitNs) {}
    }
  } else if (warp < 4) {
    // ================= rectifier warps: thread r owns token row r of every tile =================
    const int row = threadIdx.x;
    ok = warp_wait(&bars->kv_full, 0, &bars->abort_flag, status);      // z
    for (int it = 0; it < ntiles && ok; ++it) {
      const int s = it % kSlots;
      ok = warp_wait(&bars->q_full[s], (it / kSlots) & 1, &bars->abort_flag, status);
      if (!ok) break;
      float den[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        unsigned char* q = smem_al + kOffQ + (size_t)s * kTile2 + h * kHalf2 + row * 128;
        uint4 v[8];
#pragma unroll
        for (int c = 0; c < 8; ++c) v[c] = *reinterpret_cast<const uint4*>(q + ((c ^ (row & 7)) << 4));
#pragma unroll
        for (int c = 0; c < 8; ++c) {
          v[c].x = relu_bf16x2(v[c].x); v[c].y = relu_bf16x2(v[c].y); v[c].z = relu_bf16x2(v[c].z); v[c].w = relu_bf16x2(v[c].w);
          const float4 za = *reinterpret_cast<const float4*>(z_sm + 64 * h + 8 * c);
          const float4 zb = *reinterpret_cast<const float4*>(z_sm + 64 * h + 8 * c + 4);
          const float2 f0 = bf16x2_to_f2(v[c].x), f1 = bf16x2_to_f2(v[c].y), f2 = bf16x2_to_f2(v[c].z), f3 = bf16x2_to_f2(v[c].w);
          den[0] = fmaf(f0.x, za.x, fmaf(f0.y, za.y, den[0]));
          den[1] = fmaf(f1.x, za.z, fmaf(f1.y, za.w, den[1]));
          den[2] = fmaf(f2.x, zb.x, fmaf(f2.y, zb.y, den[2]));
          den[3] = fmaf(f3.x, zb.z, fmaf(f3.y, zb.w, den[3]));
        }
#pragma unroll
        for (int c = 0; c < 8; ++c) *reinterpret_cast<uint4*>(q + ((c ^ (row & 7)) << 4)) = v[c];
      }
      den_sm[s * kTok2 + row] = (den[0] + den[1]) + (den[2] + den[3]);
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      mbar_arrive(&bars->relu_done[s]);
    }
  } else {
    // ================= epilogue warps: thread (quadrant q4, lane) owns row 32 q4 + lane =================
    const int q4 = warp & 3, row = 32 * q4 + lane;
    const uint32_t lane_base = (uint32_t)(q4 << 5) << 16;
    for (int it = 0; it < ntiles; ++it) {
      const int s = it % kSlots, b = it & 1;
      // the MMAs were issued after the rectifiers had published the tile and its denominators, and are done with its slot
      ok = warp_wait(&bars->d_full[b], (it >> 1) & 1, &bars->abort_flag, status);
      if (!ok) break;
      tc_fence_after();
      const float inv = 1.f / (den_sm[s * kTok2 + row] + eps);
      unsigned char* slot = smem_al + kOffQ + (size_t)s * kTile2;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        uint32_t v0[32], v1[32];
        tmem_ld32(tmem + lane_base + b * kC + 64 * h, v0);
        tmem_ld32(tmem + lane_base + b * kC + 64 * h + 32, v1);
        tmem_wait_ld(v0);
        tmem_wait_ld(v1);
        if (h == 1) {
          tc_fence_before();
          mbar_arrive(&bars->d_empty[b]);              // the accumulator may be overwritten
        }
#pragma unroll
        for (int c = 0; c < 8; ++c) {
          const uint32_t* v = c < 4 ? v0 + 8 * c : v1 + 8 * (c - 4);
          uint4 w;
          w.x = pack_bf16(__uint_as_float(v[0]) * inv, __uint_as_float(v[1]) * inv);
          w.y = pack_bf16(__uint_as_float(v[2]) * inv, __uint_as_float(v[3]) * inv);
          w.z = pack_bf16(__uint_as_float(v[4]) * inv, __uint_as_float(v[5]) * inv);
          w.w = pack_bf16(__uint_as_float(v[6]) * inv, __uint_as_float(v[7]) * inv);
          *reinterpret_cast<uint4*>(slot + h * kHalf2 + row * 128 + ((c ^ (row & 7)) << 4)) = w;
        }
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
      if (lane == 0) {
        const int tok = t_begin + it * kTok2 + 32 * q4;
        const uint32_t src = smem + (uint32_t)kOffQ + s * kTile2 + q4 * 4096;
        if (tok < N) {                                 // rows past N inside a box are clipped by the store itself
          tma_store_3d(&mapO, src, 0, tok, bh);
          tma_store_3d(&mapO, src + kHalf2, 64, tok, bh);
        }
        asm volatile("cp.async.bulk.commit_group;" ::: "memory");
        if (it > 0) {                                  // the tile before this one: its slot may be refilled
          asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
          mbar_arrive(&bars->q_free[(it - 1) % kSlots]);
        }
      }
    }
    if (lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
    if (!ok && lane == 0) {                            // bounded time for the tensor core before tensor memory is released
      const unsigned long long t0 = globaltimer();
      while (globaltimer() - t0 < 1000000ull) {}
    }
  }
  __syncwarp();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
}

// A contiguous [BH, N, 128] bf16 tensor as (channel, token, batch*head), boxes of 64 channels x box_tok tokens
bool make_map(CUtensorMap* m, const void* ptr, int BH, int N, int box_tok) {
  EncodeFn enc = encode_fn();
  if (!enc) return false;
  const cuuint64_t dims[3] = {(cuuint64_t)kC, (cuuint64_t)N, (cuuint64_t)BH};
  const cuuint64_t strides[2] = {(cuuint64_t)kC * 2, (cuuint64_t)N * kC * 2};
  const cuuint32_t box[3] = {64, (cuuint32_t)box_tok, 1};
  const cuuint32_t estr[3] = {1, 1, 1};
  return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(ptr), dims, strides, box, estr,
             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace

bool linear_d128_supported(const LinArgs& a) {
  return a.s.dtype == JV_BF16 && a.s.D == kC && a.dwc == nullptr && !in_strided(a.s) && encode_fn() != nullptr;
}

cudaError_t launch_linear_d128(const LinArgs& a, const LinPlan& p, cudaStream_t st) {
  const jv_shape& s = a.s;
  const int N = shape_tokens(s), BH = s.B * s.H, num_sms = device_sm_count();
  int* status = device_status_ptr();
  if (!status) return cudaErrorUnknown;
  // the finished states lie over the plan's partials and states: at least (1 + 1) x 129 x 129 floats per head
  unsigned char* state = (unsigned char*)a.ws + p.off_partial;
  if ((size_t)BH * kStateBytes > p.off_hidden - p.off_partial) return cudaErrorInvalidValue;
  CUtensorMap mq, mk, mv, mo;
  if (!make_map(&mq, a.q, BH, N, kTok2) || !make_map(&mk, a.k, BH, N, kTok1) || !make_map(&mv, a.v, BH, N, kTok1) ||
      !make_map(&mo, a.o, BH, N, 32))
    return cudaErrorInvalidValue;
  static OncePerDevice opt_in;
  cudaError_t e = opt_in.run([] {
    const cudaError_t r = cudaFuncSetAttribute(lin128_state_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmem1);
    if (r != cudaSuccess) return r;
    return cudaFuncSetAttribute(lin128_apply_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmem2);
  });
  if (e != cudaSuccess) return e;

  // chunks per head: a cluster of 1, 2, 4 or 8 CTAs (the portable limit), at most one wave of two CTAs per SM, and
  // no more chunks than 64-token tiles
  const int tiles = ceil_div(N, kTok1);
  int nchunk = 1;
  while (2 * nchunk <= kMaxCluster && 2 * nchunk * BH <= 2 * num_sms && 2 * nchunk <= tiles) nchunk *= 2;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = nchunk;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(nchunk, BH);
  cfg.blockDim = dim3(kThreads1);
  cfg.dynamicSmemBytes = kSmem1;
  cfg.stream = st;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  e = cudaLaunchKernelEx(&cfg, lin128_state_kernel, mk, mv, state, status, N, ceil_div(tiles, nchunk) * kTok1);
  count_launch();
  if (e != cudaSuccess) return e;

  // one wave of one CTA per SM over (head, span of whole 128-token tiles); its set-up and first Q tiles overlap the state pass
  int nspan = num_sms / BH;
  if (nspan < 1) nspan = 1;
  const int span = ceil_div(ceil_div(N, nspan), kTok2) * kTok2;
  cudaLaunchAttribute attr2[1];
  attr2[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr2[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg2 = {};
  cfg2.gridDim = dim3(ceil_div(N, span), BH);
  cfg2.blockDim = dim3(kThreads2);
  cfg2.dynamicSmemBytes = kSmem2;
  cfg2.stream = st;
  cfg2.attrs = attr2;
  cfg2.numAttrs = 1;
  e = cudaLaunchKernelEx(&cfg2, lin128_apply_kernel, mq, mo, (const unsigned char*)state, status, N, span, a.eps);
  count_launch();
  return e;
}

}  // namespace jv
