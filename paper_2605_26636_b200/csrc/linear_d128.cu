// Linear attention (Sec. 3.2.1, Eq. 2 reordered) at head_dim 128 on the tensor cores: bf16 tensors, no convolution.
//
//   lin128_state_kernel   per (head, token chunk): KV = relu(K)^T V (tcgen05.mma, both operands as they lie in memory,
//                         ReLU in place in shared memory), z = relu(K)^T 1 in fp32.  The chunks of a head are one
//                         thread-block cluster: every CTA sends each row of its partial state to the CTA that
//                         finishes that row, which sums the chunks in order (no atomics: bit-reproducible); the finished state is written once, as the apply pass wants it: KV as a sum of kSplit bf16
//                         matrices, each already in the 128-byte-swizzled layout of its MMA operand, z in fp32.
//   lin128_apply_kernel   o = relu(q) KV / (relu(q) . z + eps) per 128-token tile: one bulk copy of the state, ReLU in place in
//                         shared memory, tcgen05.mma with the accumulator in tensor memory, TMA stores.
//
// What bounds it: HBM (K, V, Q read once, O written once: 1 KB per token and head).  At this head_dim the
// summed state is 66 KB per head: summing chunk partials in every apply CTA, as at head_dim 64, would read more than Q,
// hence the cluster reduction.  KV as three bf16 terms keeps the 24 bits of the fp32 state, so the product
// is as exact as the fp32 kernels' that served these calls before.
// Measured, 2 x 8 heads, 64 x 64 tokens: 32.6 us (67 MB) against 1330 us on the shape-generic kernels; 8 x 8 heads: 72 us
// = 3.7 TB/s.  With the state pass on mma.sync, which needs 2300 clocks of the legacy matrix path per 64 tokens (their
// copy needs 1400), and the partials read by plain remote loads it was 43 us.
#include "lin_common.cuh"

namespace jv {
namespace {

using namespace tc;
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
constexpr int kStages1 = 4;
constexpr int kReluWarps = 8;
constexpr int kThreads1 = (kReluWarps + 2) * 32;      // + TMA producer, MMA issuer
constexpr int kMaxCluster = 8;
constexpr int kLdRed = kC + 4;                        // padded row of a partial state: 16-byte accesses of 8 rows touch all banks
constexpr int kRedRows = kC + kMaxCluster;            // nchunk shares of ceil(128 / nchunk) rows
struct __align__(8) Bars1 {
  uint64_t full[kStages1], empty[kStages1];           // TMA landed / the tile's MMAs are complete
  uint64_t relu_done[kStages1];                       // 256 arrivals: K rectified
  uint64_t acc_full;                                  // all MMAs of the chunk are complete
  uint64_t red_full;                                  // the chunks' partials of this CTA's rows have landed
  uint32_t tmem_base;
  volatile uint32_t abort_flag;
};
// shared memory: ring, then this chunk's partial state over it (rows of 128 columns of KV, then z)
//                | partial states of this CTA's rows, one per chunk | z of this chunk per token group | barriers
constexpr size_t kOffRed = (size_t)kStages1 * kStage1, kOffZg = kOffRed + (size_t)kRedRows * kLdRed * sizeof(float);
constexpr size_t kOffBars1 = kOffZg + (size_t)16 * kC * sizeof(float);
constexpr size_t kSmem1 = kOffBars1 + sizeof(Bars1) + 1024;
static_assert(kSmem1 <= 232448, "shared memory of one CTA");
constexpr uint32_t kIdesc1 = idesc(128, 128, 1, 1);   // D fp32, A and B bf16, both MN-major, M = 128, N = 128

// MN-major operand of 128 columns as two swizzled halves of 64: the leading-dimension offset is the distance of the halves
__device__ __forceinline__ uint64_t smem_desc_mn128(uint32_t addr, uint32_t half_bytes) {
  return (smem_desc(addr) & ~(0x3FFFull << 16)) | ((uint64_t)(half_bytes >> 4) << 16);
}
__device__ __forceinline__ uint32_t map_rank(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}

__global__ void __launch_bounds__(kThreads1, 1)
lin128_state_kernel(const __grid_constant__ CUtensorMap mapK, const __grid_constant__ CUtensorMap mapV,
                    unsigned char* __restrict__ state, int* status, int N, int chunk_tokens) {
  extern __shared__ unsigned char smem_raw[];
  if (threadIdx.x == 32) {
    prefetch_map(&mapK);
    prefetch_map(&mapV);
  }
  unsigned char* smem_al = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  const uint32_t smem = smem_u32(smem_al);
  Bars1* bars = reinterpret_cast<Bars1*>(smem_al + kOffBars1);
  const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
  const int bh = blockIdx.y, chunk = blockIdx.x, nchunk = gridDim.x;   // the cluster is the whole grid row
  const int t_begin = min(N, chunk * chunk_tokens), t_end = min(N, t_begin + chunk_tokens);
  const int ntiles = (t_end - t_begin + kTok1 - 1) / kTok1;            // 0 for a chunk past the end

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages1; ++s) {
      mbar_init(&bars->full[s], 1);
      mbar_init(&bars->empty[s], 1);
      mbar_init(&bars->relu_done[s], kReluWarps * 32);
    }
    mbar_init(&bars->acc_full, 1);
    mbar_init(&bars->red_full, 1);
    bars->abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 0) {
    __syncwarp();
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&bars->tmem_base)), "r"(kC) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  griddep_wait();                 // what is read and written from here on may belong to the launch ahead
  // an earlier kernel gave up: no copies, no waits (but this CTA still takes part in the cluster's barriers)
  if (threadIdx.x == 0 && *reinterpret_cast<volatile int*>(status) != 0) bars->abort_flag = 1;
  __syncthreads();
  tc_fence_after();
  griddep_launch_dependents();    // (the apply pass reads Q ahead of its own wait)
  asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");   // (1) this CTA may be copied to
  const uint32_t tmem = __shfl_sync(0xffffffffu, bars->tmem_base, 0);
  bool ok = bars->abort_flag == 0;
  float* zg = reinterpret_cast<float*>(smem_al + kOffZg);              // [16 token groups][128]

  if (warp == kReluWarps) {
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
  } else if (warp == kReluWarps + 1) {
    // ================= MMA issuer: KV += relu(K)^T V, 64 tokens at a time =================
    for (int it = 0; it < ntiles && ok; ++it) {
      const int s = it % kStages1;
      ok = warp_wait(&bars->relu_done[s], (it / kStages1) & 1, &bars->abort_flag, status);
      if (!ok) break;
      tc_fence_after();
      if (elect_one()) {
        const uint64_t da = smem_desc_mn128(smem + s * kStage1, kHalf1), db = smem_desc_mn128(smem + s * kStage1 + 2 * kHalf1, kHalf1);
#pragma unroll
        for (int ks = 0; ks < kTok1 / 16; ++ks)
          mma_ss_1(tmem, desc_advance(da, ks * 2048), desc_advance(db, ks * 2048), kIdesc1, (it > 0 || ks > 0) ? 1u : 0u);
      }
      __syncwarp();
      tc_commit(&bars->empty[s]);
    }
    if (ok && ntiles > 0) tc_commit(&bars->acc_full);
    if (!ok && lane == 0) {                                 // bounded time for the tensor core before tensor memory is released
      const unsigned long long t0 = globaltimer();
      while (globaltimer() - t0 < 1000000ull) {}
    }
  } else {
    // ================= rectifier warps: thread owns 16-byte chunk cc of tokens 4 tg .. 4 tg + 3 of every tile: ReLU in
    // place, and z of its eight channels exactly in fp32 =================
    const int cc = threadIdx.x & 15, tg = threadIdx.x >> 4;
    float z[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) z[e] = 0.f;
    for (int it = 0; it < ntiles && ok; ++it) {
      const int s = it % kStages1;
      ok = warp_wait(&bars->full[s], (it / kStages1) & 1, &bars->abort_flag, status);
      if (!ok) break;
      unsigned char* kt = smem_al + (size_t)s * kStage1 + (cc >> 3) * kHalf1;
      uint4 x[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) x[j] = *reinterpret_cast<const uint4*>(kt + tile_off(4 * tg + j, cc & 7));
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        x[j].x = relu_bf16x2(x[j].x); x[j].y = relu_bf16x2(x[j].y); x[j].z = relu_bf16x2(x[j].z); x[j].w = relu_bf16x2(x[j].w);
        *reinterpret_cast<uint4*>(kt + tile_off(4 * tg + j, cc & 7)) = x[j];
        const float2 f0 = bf16x2_to_f2(x[j].x), f1 = bf16x2_to_f2(x[j].y), f2 = bf16x2_to_f2(x[j].z), f3 = bf16x2_to_f2(x[j].w);
        z[0] += f0.x; z[1] += f0.y; z[2] += f1.x; z[3] += f1.y;
        z[4] += f2.x; z[5] += f2.y; z[6] += f3.x; z[7] += f3.y;
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      mbar_arrive(&bars->relu_done[s]);
    }
    *reinterpret_cast<float4*>(zg + tg * kC + 8 * cc) = make_float4(z[0], z[1], z[2], z[3]);
    *reinterpret_cast<float4*>(zg + tg * kC + 8 * cc + 4) = make_float4(z[4], z[5], z[6], z[7]);
    if (ok && ntiles > 0) ok = warp_wait(&bars->acc_full, 0, &bars->abort_flag, status);
    tc_fence_after();
  }
  __syncthreads();
  // The partial state goes to shared memory (over the ring: its copies have landed and its MMAs are complete), thread
  // (quadrant q4, lane) holding row 32 q4 + lane, warps 0-3 its columns 0-63 and z, warps 4-7 columns 64-127; from there one
  // bulk copy takes every CTA of the cluster the rows that it finishes.  (Stored to the other CTAs straight from
  // the registers, 16 bytes of a row per lane, the 64 KB took 6000 clocks.)
  const int share = (kC + nchunk - 1) / nchunk;
  if (warp < kReluWarps) {
    const int q4 = warp & 3, h = warp >> 2, row = 32 * q4 + lane;
    float* dst = reinterpret_cast<float*>(smem_al) + row * kLdRed + 64 * h;
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      uint32_t v[32];
      if (ntiles > 0) {
        tmem_ld32(tmem + ((uint32_t)(q4 << 5) << 16) + 64 * h + 32 * j, v);
        tmem_wait_ld(v);
      } else {
#pragma unroll
        for (int i = 0; i < 32; ++i) v[i] = 0u;
      }
#pragma unroll
      for (int i = 0; i < 32; i += 4)
        *reinterpret_cast<uint4*>(dst + 32 * j + i) = make_uint4(v[i], v[i + 1], v[i + 2], v[i + 3]);
    }
    if (h == 0) {
      float z = 0.f;
#pragma unroll
      for (int g = 0; g < 16; ++g) z += zg[g * kC + row];
      dst[kC] = z;
    }
    tc_fence_before();
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  __syncthreads();
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");     // (1)
  const int row0 = chunk * share, rows = max(0, min(share, kC - row0));
  if (warp == 0 && elect_one()) {
    if (rows > 0) mbar_expect_tx(&bars->red_full, (uint32_t)(nchunk * rows * kLdRed * 4));
    for (int c = 0; c < nchunk; ++c) {
      const int n = min(share, kC - c * share);
      if (n > 0)
        asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                     ::"r"(map_rank(smem + (uint32_t)kOffRed + (uint32_t)(chunk * share * kLdRed * 4), c)),
                       "r"(smem + (uint32_t)(c * share * kLdRed * 4)), "r"((uint32_t)(n * kLdRed * 4)),
                       "r"(map_rank(smem_u32(&bars->red_full), c)) : "memory");
    }
  }
  __syncwarp();
  if (rows > 0) {
    // Every CTA sends, also one that gave up, and none may leave while copies into its shared memory are on their way: this wait
    // is bounded by time alone, whatever the abort flag says.
    const unsigned long long t0 = globaltimer();
    bool landed;
    while (!(landed = mbar_try(&bars->red_full, 0)) && globaltimer() - t0 < kWaitLimitNs) {}
    if (!landed) atomicOr(status, kStatusTimeout);
  }
  asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");   // (2) received: the senders may leave
  // this CTA's rows: the chunks' partials summed in chunk order, eight columns per thread and step
  const float* red = reinterpret_cast<const float*>(smem_al + kOffRed);
  unsigned char* st = state + (size_t)bh * kStateBytes;
  for (int i = threadIdx.x; i < rows * (kC / 8); i += kThreads1) {
    const int r = i / (kC / 8), c8 = i % (kC / 8);
    float x[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) x[e] = 0.f;
    for (int c = 0; c < nchunk; ++c) {
      const float* src = red + (c * share + r) * kLdRed + 8 * c8;
      const float4 lo = *reinterpret_cast<const float4*>(src), hi = *reinterpret_cast<const float4*>(src + 4);
      x[0] += lo.x; x[1] += lo.y; x[2] += lo.z; x[3] += lo.w;
      x[4] += hi.x; x[5] += hi.y; x[6] += hi.z; x[7] += hi.w;
    }
#pragma unroll
    for (int s = 0; s < kSplit; ++s) {                      // the bf16 nearest to what the terms before it left over
      uint32_t w[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        w[e] = pack_bf16(x[2 * e], x[2 * e + 1]);
        const float2 f = bf16x2_to_f2(w[e]);
        x[2 * e] = isinf(f.x) ? 0.f : x[2 * e] - f.x;       // (infinity leaves nothing over: inf - inf would be NaN)
        x[2 * e + 1] = isinf(f.y) ? 0.f : x[2 * e + 1] - f.y;
      }
      *reinterpret_cast<uint4*>(st + (size_t)(2 * s + (c8 >> 3)) * kKvHalf + tile_off(row0 + r, c8 & 7)) = make_uint4(w[0], w[1], w[2], w[3]);
    }
  }
  for (int i = threadIdx.x; i < rows; i += kThreads1) {
    float z = 0.f;
    for (int c = 0; c < nchunk; ++c) z += red[(c * share + i) * kLdRed + kC];
    reinterpret_cast<float*>(st + kKvBytes)[row0 + i] = z;
  }
  tc_fence_after();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kC) : "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");     // (2)
}

// ---- apply pass ---------------------------------------------------------------------
constexpr int kTok2 = 128;                            // tokens per tile
constexpr int kHalf2 = kTok2 * 128;                   // 128 tokens x 64 channels: 16 KB
constexpr int kTile2 = 2 * kHalf2;
constexpr int kSlots = 3;                             // Q tiles; a slot becomes its tile's output staging
constexpr int kThreads2 = 320;                        // 4 rectifier warps, MMA issuer, 4 epilogue warps, TMA producer
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
constexpr uint32_t kIdesc2 = idesc(128, 128, 1);      // D fp32, A and B bf16, B MN-major, M = 128, N = 128

__global__ void __launch_bounds__(kThreads2, 1)
lin128_apply_kernel(const __grid_constant__ CUtensorMap mapQ, const __grid_constant__ CUtensorMap mapO,
                    const unsigned char* __restrict__ state, int* status, int N, int span_tokens, float eps) {
  extern __shared__ unsigned char smem_raw[];
  if (threadIdx.x == 32) {
    prefetch_map(&mapQ);
    prefetch_map(&mapO);
  }
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
  griddep_launch_dependents();
  const uint32_t tmem = __shfl_sync(0xffffffffu, bars->tmem_base, 0);
  bool ok = true;

  if (warp == 9) {
    // ================= TMA producer =================
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
                     ::"r"(smem_u32(z_sm)), "l"(state + (size_t)bh * kStateBytes + kKvBytes), "r"(kC * 4),
                       "r"(smem_u32(&bars->kv_full)) : "memory");
        asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                     ::"r"(smem), "l"(state + (size_t)bh * kStateBytes), "r"(kKvBytes), "r"(smem_u32(&bars->kv_full)) : "memory");
      }
      __syncwarp();
    }
    for (int it = kSlots; it < ntiles && ok; ++it) {
      ok = warp_wait(&bars->q_free[it % kSlots], ((it / kSlots) - 1) & 1, &bars->abort_flag, status);
      if (ok) load_tile(it);
    }
    if (!ok && lane == 0) {                            // let the copies in flight land before the CTA leaves
      const unsigned long long t0 = globaltimer();
      for (int g = max(0, issued - kSlots); g < issued; ++g)
        while (!mbar_try(&bars->q_full[g % kSlots], (g / kSlots) & 1) && globaltimer() - t0 < kWaitLimitNs) {}
      while (kv_issued && !mbar_try(&bars->kv_full, 0) && globaltimer() - t0 < kWaitLimitNs) {}
    }
  } else if (warp == 4) {
    // ================= MMA issuer =================
    ok = warp_wait(&bars->kv_full, 0, &bars->abort_flag, status);
    for (int it = 0; it < ntiles && ok; ++it) {
      const int s = it % kSlots, b = it & 1;
      ok = warp_wait(&bars->relu_done[s], (it / kSlots) & 1, &bars->abort_flag, status);
      if (ok && it >= 2) ok = warp_wait(&bars->d_empty[b], ((it >> 1) - 1) & 1, &bars->abort_flag, status);
      if (!ok) break;
      tc_fence_after();
      if (elect_one()) {
        const uint64_t da = smem_desc(smem + (uint32_t)kOffQ + s * kTile2);
#pragma unroll
        for (int x = 0; x < kSplit; ++x) {
          const uint64_t db = smem_desc_mn128(smem + 2 * x * kKvHalf, kKvHalf);
#pragma unroll
          for (int ks = 0; ks < kC / 16; ++ks)
            mma_ss_1(tmem + b * kC, desc_advance(da, (ks >> 2) * kHalf2 + (ks & 3) * 32), desc_advance(db, ks * 2048), kIdesc2,
                     (x > 0 || ks > 0) ? 1u : 0u);
        }
      }
      __syncwarp();
      tc_commit(&bars->d_full[b]);
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

  // chunks per head: a cluster of up to 8 CTAs (the portable limit), one CTA per SM over all heads
  const int tiles = ceil_div(N, kTok1);
  int nchunk = num_sms / BH;
  if (nchunk > kMaxCluster) nchunk = kMaxCluster;
  if (nchunk > tiles) nchunk = tiles;
  if (nchunk < 1) nchunk = 1;
  e = launch_cluster(true, lin128_state_kernel, nchunk, dim3(nchunk, BH), kThreads1, kSmem1, st, mk, mv, state, status, N,
                                  ceil_div(tiles, nchunk) * kTok1);
  if (e != cudaSuccess) return e;

  // one wave of one CTA per SM over (head, span of whole 128-token tiles); its set-up and first Q tiles overlap the state pass
  int nspan = num_sms / BH;
  if (nspan < 1) nspan = 1;
  const int span = ceil_div(ceil_div(N, nspan), kTok2) * kTok2;
  return launch_programmatic(lin128_apply_kernel, dim3(ceil_div(N, span), BH), kThreads2, kSmem2, st, mq, mo, (const unsigned char*)state,
                             status, N, span, a.eps);
}

}  // namespace jv
