// The linear projections either side of a token mixer (the inherited W_Q, W_K, W_V and W_O
// of every block, Sec. 3.2.4) as tcgen05 GEMMs that read and write the mixers' [B, H, N, 64]
// layout directly, so that no transpose pass runs between the projection and the mixer.
//
//   qkv:  x [B, N, C] (C = H * 64)  times  w [3C, C]^T  ->  q, k, v [B, H, N, 64]
//         output feature f = which * C + h * 64 + e  (which: 0 = q, 1 = k, 2 = v)
//   out:  o [B, H, N, 64]  times  w [C, C]^T  ->  y [B, N, C]
//         input feature h * 64 + e: one K block of 64 is one head of o
//
// One persistent CTA per SM loops over output tiles of 128 tokens x 256 features, or a pair of CTAs over tiles of 2 x 128 x 256
// (template parameter kCtas; feature tile fastest, so what runs together shares its token tiles in L2 and the weights stay
// L2-resident).  In a pair tcgen05.mma runs in its two-SM form (cta_group::2, M 256, N 256): each CTA holds one of the two token
// tiles, which need not be neighbours, half of the tile's weights, and the accumulator rows of its own tokens.
// What bounds a tile of one CTA is not the tensor pipe but shared memory: a K block of 64 is 48 KB written by the copies
// and 48 KB read by the MMAs, 768 clocks for 512 clocks of MMA; with the weights shared by two CTAs it is 32 + 32 KB.
// Measured (2 x 8192 tokens, 768 -> 2304 / 8 x 4096 tokens, 1024 -> 3072 features, in turn): 44.4 / 140 us = 1307 / 1475 TF in pairs, 48.2 / 157
// singly, in short runs; 51.5 / 160 and 55.4 / 184 in a long loop at the power cap.  With four epilogue warps instead of eight and the bias fetched
// after the accumulator (single CTAs, another run) 53.4 / 152, when this form took 49.7 / 153.
// Warp roles (both CTAs of a pair):
//   warp 0      TMA producer: A (128 tokens x 64) and (half of) B (256 features x 64) through a ring of 4 (5) stages; the
//               copies of both CTAs report to the leader's barrier
//   warp 1      (leader, the even CTA) MMA issuer: 4 x tcgen05.mma K16 per stage into one of two
//               accumulators in tensor memory (2 x 256 columns in each CTA); its commits arrive in both CTAs
//   warps 4-11  epilogue of the other accumulator, two warps per tensor-memory quadrant: tensor memory -> registers, + bias, bf16,
//               swizzled staging in shared memory, one TMA store per warp and 64-feature block
// Token tiles never cross a batch element: rows past N are zero-filled on load and clipped on
// store by TMA; feature blocks past the last one are skipped.
//
// Every mbarrier wait is bounded; a wait that runs out sets the device status word and the
// CTA's abort flag, and every role falls through to the teardown that frees tensor memory.
#include "tc_common.cuh"

namespace jv {
namespace {

using namespace tc;

constexpr int kD = 64;                       // head_dim = K block = feature block
constexpr int kBM = 128;                     // tokens per CTA and tile
constexpr int kBN = 256;                     // features per tile
constexpr int kABytes = kBM * kD * 2;        // 16 KB
constexpr int kEpiWarps = 8;                 // two per tensor-memory quadrant, each with half of the tile's features
constexpr int kThreads = (4 + kEpiWarps) * 32;
constexpr uint32_t kTmemCols = 512;
constexpr int kStagingBytes = 32 * kD * 2;   // one warp's 32 tokens x 64 features
constexpr int kMaxStages = 5;

// kCtas: CTAs per tile, 1 or 2 (a pair)
template <int kCtas>
struct Layout {
  static constexpr int kBBytes = kBN / kCtas * kD * 2;             // this CTA's part of the features
  static constexpr int kStageBytes = kABytes + kBBytes;
  static constexpr int kStages = kCtas == 2 ? 5 : 4;
  static constexpr int kBufs = kCtas == 2 ? 2 : 1;                 // staging buffers per epilogue warp
  static constexpr size_t kTiles = (size_t)kStages * kStageBytes + (size_t)kEpiWarps * kBufs * kStagingBytes;
};
struct __align__(8) Barriers {
  uint64_t full[kMaxStages], empty[kMaxStages];    // full, acc_empty: the leader's count for the pair
  uint64_t acc_full[2], acc_empty[2];
  uint64_t drain;
  uint32_t tmem_base;
  volatile uint32_t abort_flag;
};
template <int kCtas>
constexpr size_t smem_bytes() { return Layout<kCtas>::kTiles + sizeof(Barriers) + 1024; }
static_assert(smem_bytes<1>() <= 232448 && smem_bytes<2>() <= 232448, "shared memory of one CTA");

struct ProjParams {
  const float* bias;       // [features] or nullptr
  int bias_vec;            // bias is 16-byte aligned
  int* status;
  int tiles_m_per_batch;   // ceil(N / 128)
  int tiles_n;             // ceil(features / 256)
  int tiles_m;             // B * tiles_m_per_batch
  int total_tiles;         // ceil(tiles_m / 2) * tiles_n: tiles of a pair of CTAs
  int kblocks;             // C / 64
  int H;                   // heads
  int fblocks;             // features / 64
  int N;                   // tokens per batch element
  int silu;                // 1: x / (1 + exp(-x)) on the result (the kernel generator's hidden layer)
  int out_f16;             // 1: the result is stored as fp16 instead of bf16 (same size; the generator's intermediates)
  uint32_t idesc;          // instruction descriptor: bf16 or fp16 operands
};

// Instruction descriptors: M128 (one CTA) or M256 (a pair) x N256, both operands K-major; bf16 operands, or fp16 ones (format 0 in both fields)
constexpr uint32_t kIdesc1 = idesc(kBM, kBN, 0), kIdesc2 = idesc(2 * kBM, kBN, 0);
constexpr uint32_t kIdescF16Mask = ~((1u << 7) | (1u << 10));
__device__ __forceinline__ uint32_t pack_f16(float lo, float hi) {
  uint32_t r;
  asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
  return r;
}

struct Tile {
  int b, tok0, f0;   // batch element, this CTA's first token (N: it has no tile, an odd one out), first feature
};
template <int kCtas>
__device__ __forceinline__ Tile decode_tile(const ProjParams& p, int i, int rank) {
  const int tn = i % p.tiles_n, m = kCtas * (i / p.tiles_n) + rank;
  if (m >= p.tiles_m) return Tile{0, p.N, tn * kBN};
  const int tm = m % p.tiles_m_per_batch, b = m / p.tiles_m_per_batch;
  return Tile{b, tm * kBM, tn * kBN};
}

// ---- one CTA, or the two-SM forms, whose addresses are of the cluster's shared memory -----------------------------------
__device__ __forceinline__ uint32_t map_rank(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void tma_load_3d_pair(uint32_t dst, const CUtensorMap* map, uint32_t bar, int c0, int c1, int c2) {
  asm volatile("cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];"
               ::"r"(dst), "l"(map), "r"(bar), "r"(c0), "r"(c1), "r"(c2) : "memory");
}
__device__ __forceinline__ void tma_load_2d_pair(uint32_t dst, const CUtensorMap* map, uint32_t bar, int c0, int c1) {
  asm volatile("cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
               ::"r"(dst), "l"(map), "r"(bar), "r"(c0), "r"(c1) : "memory");
}
__device__ __forceinline__ void mma_ss_pair(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n}\n"
      ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(acc) : "memory");
}
// arrives on the barrier (at this offset in both CTAs of a pair) once the MMAs issued so far are complete
template <bool kPair>
__device__ __forceinline__ void commit(uint64_t* bar) {
  if (!kPair) tc_commit(bar);
  else if (elect_one())
    asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
                 ::"r"(smem_u32(bar)), "h"((uint16_t)3) : "memory");
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }

// kQKV: A = x as (C, N, B), outputs q, k, v as (64, N, B*H); else A = o as (64, N, B*H),
// output y as (C, N, B).  B (the weights) is (C, features) in both.
template <bool kQKV, int kCtas>
__global__ void __launch_bounds__(kThreads, 1)
proj_tc_kernel(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapB,
               const __grid_constant__ CUtensorMap mapD0, const __grid_constant__ CUtensorMap mapD1,
               const __grid_constant__ CUtensorMap mapD2, const ProjParams p) {
  extern __shared__ unsigned char smem_raw[];
  if (threadIdx.x == 32) {
    prefetch_map(&mapA);
    prefetch_map(&mapB);
    prefetch_map(&mapD0);
  }
  // 1024-byte alignment by an offset from the array itself, so that accesses stay shared-space loads and stores
  unsigned char* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  using L = Layout<kCtas>;
  constexpr int kStages = L::kStages, kStageBytes = L::kStageBytes, kBufs = L::kBufs;
  constexpr bool kPair = kCtas == 2;
  Barriers* bar = reinterpret_cast<Barriers*>(smem + L::kTiles);
  const uint32_t sRing = smem_u32(smem), sStage = sRing + kStages * kStageBytes;

  const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;

  const int rank = kPair ? blockIdx.x & 1 : 0;   // in the pair: 0 leads

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(&bar->full[s], 1);
      mbar_init(&bar->empty[s], 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(&bar->acc_full[a], 1);
      mbar_init(&bar->acc_empty[a], kCtas * kEpiWarps);      // lane 0 of each epilogue warp
    }
    mbar_init(&bar->drain, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 0) {
    __syncwarp();
    if (kPair) {
      asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&bar->tmem_base)),
                   "r"(kTmemCols) : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    } else {
      asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&bar->tmem_base)),
                   "r"(kTmemCols) : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
  }
  griddep_wait();                            // what is read and written from here on may belong to the launch ahead
  // a timeout flagged earlier (by any CTA or launch) makes the rest leave at once: as the leader sees it, for both CTAs
  if (threadIdx.x == 0) bar->abort_flag = *reinterpret_cast<volatile int*>(p.status) != 0;
  uint32_t gave_up;
  if (kPair) {
    __syncwarp();
    cluster_arrive();
    cluster_wait();
    asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(gave_up) : "r"(map_rank(smem_u32((const void*)&bar->abort_flag), 0)) : "memory");
    cluster_arrive();                        // (the leader may not leave or raise its flag before the other CTA has read it)
    cluster_wait();
  } else {
    __syncthreads();
    gave_up = bar->abort_flag;
    __syncthreads();
  }
  if (threadIdx.x == 0) bar->abort_flag = 0;
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = __shfl_sync(0xffffffffu, bar->tmem_base, 0);
  griddep_launch_dependents();
  auto free_tmem = [&]() {
    if (kPair) asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
    else asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
  };
  if (gave_up) {
    if (warp == 0) free_tmem();
    return;
  }

  const int tile0 = blockIdx.x / kCtas, tile_step = gridDim.x / kCtas;

  if (warp == 0) {
    // ================= TMA producer =================
    bool ok = true;
    int s = 0, issued = 0;
    uint32_t par = 1;
    for (int i = tile0; i < p.total_tiles && ok; i += tile_step) {
      const Tile t = decode_tile<kCtas>(p, i, rank);
      for (int kb = 0; kb < p.kblocks; ++kb) {
        ok = warp_wait(&bar->empty[s], par, &bar->abort_flag, p.status);
        if (!ok) break;
        if (elect_one()) {
          const uint32_t dst = sRing + s * kStageBytes;
          const int a0 = kQKV ? kb * kD : 0, a2 = kQKV ? t.b : t.b * p.H + kb % p.H;   // (more K blocks than planes: A repeats)
          if (rank == 0) mbar_expect_tx(&bar->full[s], kCtas * kStageBytes);           // what both CTAs' copies bring
          if (kPair) {
            const uint32_t full = map_rank(smem_u32(&bar->full[s]), 0);
            tma_load_3d_pair(dst, &mapA, full, a0, t.tok0, a2);
            tma_load_2d_pair(dst + kABytes, &mapB, full, kb * kD, t.f0 + rank * (kBN / 2));
          } else {
            tma_load_3d(dst, &mapA, &bar->full[s], a0, t.tok0, a2);
            tma_load_2d(dst + kABytes, &mapB, &bar->full[s], kb * kD, t.f0);
          }
        }
        __syncwarp();
        ++issued;
        if (++s == kStages) { s = 0; par ^= 1; }
      }
    }
    if (!ok && lane == 0) {
      // let the copies still in flight land before the CTA leaves (bounded by the same limit; the leader's barriers tell)
      const unsigned long long t0 = globaltimer();
      for (int g = max(0, issued - kStages); g < issued && rank == 0; ++g)
        while (!mbar_try(&bar->full[g % kStages], (g / kStages) & 1) && globaltimer() - t0 < kWaitLimitNs) {}
      while (rank != 0 && globaltimer() - t0 < 1000000ull) {}
    }
  } else if (warp == 1 && rank == 0) {
    // ================= MMA issuer (of the pair) =================
    bool ok = true;
    int s = 0, n = 0;
    uint32_t ph = 0;
    for (int i = tile0; i < p.total_tiles && ok; i += tile_step, ++n) {
      const int a = n & 1;
      ok = warp_wait(&bar->acc_empty[a], ((n >> 1) & 1) ^ 1, &bar->abort_flag, p.status);   // epilogue has read tile n - 2
      if (!ok) break;
      tc_fence_after();
      const uint32_t d = tmem + a * kBN;
      for (int kb = 0; kb < p.kblocks; ++kb) {
        ok = warp_wait(&bar->full[s], ph, &bar->abort_flag, p.status);
        if (!ok) break;
        tc_fence_after();
        const uint32_t sa = sRing + s * kStageBytes, sb = sa + kABytes;
        if (elect_one()) {
          const uint64_t da = smem_desc(sa), db = smem_desc(sb);
#pragma unroll
          for (int ks = 0; ks < kD / 16; ++ks)
            if (kPair) mma_ss_pair(d, desc_advance(da, ks * 32), desc_advance(db, ks * 32), p.idesc, (kb > 0 || ks > 0) ? 1u : 0u);
            else mma_ss_1(d, desc_advance(da, ks * 32), desc_advance(db, ks * 32), p.idesc, (kb > 0 || ks > 0) ? 1u : 0u);
        }
        __syncwarp();
        commit<kPair>(&bar->empty[s]);
        if (++s == kStages) { s = 0; ph ^= 1; }
      }
      if (ok) commit<kPair>(&bar->acc_full[a]);
    }
    // every MMA issued so far must have retired before tensor memory is released
    commit<kPair>(&bar->drain);
    if (lane == 0) {
      const unsigned long long t0 = globaltimer();
      while (!mbar_try(&bar->drain, 0) && globaltimer() - t0 < kWaitLimitNs) {}
    }
    __syncwarp();
  } else if (warp >= 4) {
    // ================= epilogue: one thread per token row =================
    const int q4 = warp & 3, half = (warp - 4) >> 2;   // the warp's tensor-memory quadrant; which half of the tile's features
    const uint32_t lane_base = (uint32_t)(q4 << 5) << 16;
    unsigned char* stage_ptr = smem + kStages * kStageBytes + (warp - 4) * kBufs * kStagingBytes;
    const uint32_t stage_u32 = sStage + (warp - 4) * kBufs * kStagingBytes;
    bool ok = true;
    int n = 0, nstore = 0;
    for (int i = tile0; i < p.total_tiles && ok; i += tile_step, ++n) {
      const Tile t = decode_tile<kCtas>(p, i, rank);
      const int a = n & 1;
      ok = warp_wait(&bar->acc_full[a], (n >> 1) & 1, &bar->abort_flag, p.status);
      if (!ok) break;
      tc_fence_after();
      const int tok = t.tok0 + 32 * q4;
#pragma unroll 1
      for (int j = 2 * half; j < 2 * half + 2; ++j) {
        const int fb = t.f0 / kD + j;
        if (fb >= p.fblocks || tok >= p.N) break;   // no such features / none of this warp's rows exists
        uint32_t ob[32];
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          uint32_t v[32];
          tmem_ld32(tmem + lane_base + a * kBN + j * kD + c * 32, v);
          float4 bb[8];                       // the bias, on its way beside the accumulator (coherent loads: the launch ahead may write it)
#pragma unroll
          for (int i4 = 0; i4 < 8; ++i4) {
            const float* bp = p.bias + fb * kD + c * 32 + 4 * i4;
            bb[i4] = !p.bias ? make_float4(0.f, 0.f, 0.f, 0.f)
                     : p.bias_vec ? *reinterpret_cast<const float4*>(bp)
                                  : make_float4(bp[0], bp[1], bp[2], bp[3]);
          }
          tmem_wait_ld(v);
#pragma unroll
          for (int i4 = 0; i4 < 8; ++i4) {
            v[4 * i4] = __float_as_uint(__uint_as_float(v[4 * i4]) + bb[i4].x);
            v[4 * i4 + 1] = __float_as_uint(__uint_as_float(v[4 * i4 + 1]) + bb[i4].y);
            v[4 * i4 + 2] = __float_as_uint(__uint_as_float(v[4 * i4 + 2]) + bb[i4].z);
            v[4 * i4 + 3] = __float_as_uint(__uint_as_float(v[4 * i4 + 3]) + bb[i4].w);
          }
          if (p.silu) {
#pragma unroll
            for (int i2 = 0; i2 < 32; ++i2) {
              const float z = __uint_as_float(v[i2]);
              v[i2] = __float_as_uint(z / (1.f + __expf(-z)));
            }
          }
#pragma unroll
          for (int i2 = 0; i2 < 16; ++i2)
            ob[16 * c + i2] = p.out_f16 ? pack_f16(__uint_as_float(v[2 * i2]), __uint_as_float(v[2 * i2 + 1]))
                                        : pack_bf16(__uint_as_float(v[2 * i2]), __uint_as_float(v[2 * i2 + 1]));
        }
        // the store that last used this staging buffer must have finished reading it
        const int sbuf = kBufs == 2 ? nstore & 1 : 0;
        if (lane == 0) asm volatile("cp.async.bulk.wait_group.read %0;" ::"n"(kBufs - 1) : "memory");
        __syncwarp();
#pragma unroll
        for (int c = 0; c < 8; ++c)     // 16-byte chunk c of this row, at its 128-byte-swizzle position
          *reinterpret_cast<uint4*>(stage_ptr + sbuf * kStagingBytes + lane * 128 + ((c ^ (lane & 7)) << 4)) =
              make_uint4(ob[4 * c], ob[4 * c + 1], ob[4 * c + 2], ob[4 * c + 3]);
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
        if (lane == 0) {
          const uint32_t src = stage_u32 + sbuf * kStagingBytes;
          if (kQKV) {
            const int which = fb / p.H, h = fb - which * p.H;
            const CUtensorMap* m = which == 0 ? &mapD0 : which == 1 ? &mapD1 : &mapD2;
            tma_store_3d(m, src, 0, tok, t.b * p.H + h);
          } else {
            tma_store_3d(&mapD0, src, fb * kD, tok, t.b);
          }
          asm volatile("cp.async.bulk.commit_group;" ::: "memory");
        }
        ++nstore;
      }
      // this accumulator may be overwritten once all epilogue warps have read it
      tc_fence_before();
      __syncwarp();
      if (lane == 0) {
        if (kPair)
          asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(map_rank(smem_u32(&bar->acc_empty[a]), 0)) : "memory");
        else
          mbar_arrive(&bar->acc_empty[a]);
      }
    }
    if (lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
  }

  // ================= common teardown =================
  // The leader's commits arrive in the other CTA's shared memory, too: that one stays until the last of them has
  // (bounded by time; the leader has waited for its own).
  if (kPair && rank != 0 && warp == 4 && lane == 0) {
    const unsigned long long t0 = globaltimer();
    while (!mbar_try(&bar->drain, 0) && globaltimer() - t0 < kWaitLimitNs) {}
  }
  __syncwarp();
  tc_fence_before();
  if (kPair) {
    cluster_arrive();                        // neither CTA leaves, or frees tensor memory, while the other's commits and arrivals may come
    cluster_wait();
  } else {
    __syncthreads();
  }
  tc_fence_after();
  if (warp == 0) free_tmem();
}

// ---- host side ----------------------------------------------------------------------
// bf16 tensor (inner, rows, outer), contiguous, with a box of (64, box_rows, 1)
bool map3(CUtensorMap* m, const void* ptr, uint64_t inner, uint64_t rows, uint64_t outer, uint32_t box_rows) {
  const cuuint64_t dims[3] = {inner, rows, outer};
  const cuuint64_t strides[2] = {inner * 2, inner * rows * 2};
  const cuuint32_t box[3] = {(cuuint32_t)kD, box_rows, 1};
  const cuuint32_t estr[3] = {1, 1, 1};
  return encode_fn()(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(ptr), dims, strides, box, estr,
                     CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                     CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}
// bf16 matrix (inner, rows), contiguous, with a box of (64, box_rows)
bool map2(CUtensorMap* m, const void* ptr, uint64_t inner, uint64_t rows, uint32_t box_rows) {
  const cuuint64_t dims[2] = {inner, rows};
  const cuuint64_t strides[1] = {inner * 2};
  const cuuint32_t box[2] = {(cuuint32_t)kD, box_rows};
  const cuuint32_t estr[2] = {1, 1};
  return encode_fn()(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(ptr), dims, strides, box, estr,
                     CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                     CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace

bool proj_tc_available() { return encode_fn() != nullptr; }

namespace {

template <bool kQKV, int kCtas>
cudaError_t launch(const CUtensorMap& ma, const CUtensorMap& mb, const CUtensorMap& md0, const CUtensorMap& md1, const CUtensorMap& md2,
                   const ProjParams& p, cudaStream_t st) {
  static OncePerDevice opt_in;   // > 48 KB of dynamic shared memory: a per-device function attribute
  const cudaError_t e = opt_in.run([] {
    return cudaFuncSetAttribute(proj_tc_kernel<kQKV, kCtas>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_bytes<kCtas>());
  });
  if (e != cudaSuccess) return e;
  const int slots = device_sm_count() / kCtas;
  const dim3 grid(kCtas * (p.total_tiles < slots ? p.total_tiles : slots));
  if (kCtas == 1) return launch_programmatic(proj_tc_kernel<kQKV, kCtas>, grid, kThreads, smem_bytes<kCtas>(), st, ma, mb, md0, md1, md2, p);
  return launch_cluster(true, proj_tc_kernel<kQKV, kCtas>, kCtas, grid, kThreads, smem_bytes<kCtas>(), st, ma, mb, md0, md1, md2, p);
}

// Pairs of CTAs where every pair has three tiles or more: a pair takes 2 us longer to start (cluster launch, two cluster
// barriers) and a tile of it is a tenth faster or more.  Measured in turn in long loops, single / pair: 24 tiles of a pair 8.9 / 10.0 us, 72: 9.6 / 10.7,
// 96: 13.6 / 14.2, 192: 18.5 / 18.5 and (16 K blocks) 22.5 / 21.6, 288: 23.9 / 23.9 and (24) 48.5 / 45.2, 576: 55.4 / 51.5, 512 (16): 66.8 / 61.0, 1536:
// 184 / 160.
bool pair_tiles(int64_t tiles_m, int tiles_n) {
  return (tiles_m + 1) / 2 * tiles_n >= 3 * (device_sm_count() / 2);
}

// Fills in what depends on the problem's size; false if there are too many tiles.
bool plan(ProjParams& p, bool pair, int B, int N, int features, int kblocks, bool f16) {
  const int ctas = pair ? 2 : 1;
  p.tiles_m_per_batch = ceil_div(N, kBM);
  p.tiles_n = ceil_div(features, kBN);
  p.tiles_m = B * p.tiles_m_per_batch;
  const int64_t total = (int64_t)ceil_div(p.tiles_m, ctas) * p.tiles_n;
  p.total_tiles = (int)total;
  p.kblocks = kblocks;
  p.fblocks = features / kD;
  p.N = N;
  p.idesc = (pair ? kIdesc2 : kIdesc1) & (f16 ? kIdescF16Mask : ~0u);
  return total <= 0x7fffffffll;
}

}  // namespace

// The kernel on its own terms (see common.cuh).  kQKV of the kernel means "A is [B, N, K]" for the loads
// and "D is planes" for the stores, which go together in the two projections; the other two
// combinations are reached through the plane count: with one K block per "head" ... the generator's
// GEMMs need A planes -> D rows (the out form, as it is) and A rows -> D planes (the qkv form with
// every feature block a plane of its own: H := F / 64, so that "which" is always 0).
cudaError_t launch_proj_gemm(bool planes_in, bool planes_out, const void* A, const void* W, const float* bias, void* D, int B,
                             int N, int kblocks, int a_planes, int F, bool silu, bool f16_in, bool f16_out, int* status,
                             cudaStream_t st) {
  if (!encode_fn() || planes_in == planes_out || F % kD != 0) return cudaErrorNotSupported;
  const uint64_t K = (uint64_t)kblocks * kD;
  const bool pair = pair_tiles((int64_t)B * ceil_div(N, kBM), ceil_div(F, kBN));
  CUtensorMap ma, mb, md;
  bool ok = map2(&mb, W, K, (uint64_t)F, pair ? kBN / 2 : kBN);
  if (planes_in) ok = ok && map3(&ma, A, kD, (uint64_t)N, (uint64_t)B * a_planes, kBM) && map3(&md, D, (uint64_t)F, (uint64_t)N, (uint64_t)B, 32);
  else ok = ok && map3(&ma, A, K, (uint64_t)N, (uint64_t)B, kBM) && map3(&md, D, kD, (uint64_t)N, (uint64_t)B * (F / kD), 32);
  ProjParams p;
  if (!ok || !plan(p, pair, B, N, F, kblocks, f16_in)) return cudaErrorInvalidValue;
  p.bias = bias;
  p.bias_vec = ((uintptr_t)bias & 15) == 0;
  p.status = status;
  p.H = planes_in ? a_planes : F / kD;
  p.silu = silu ? 1 : 0;
  p.out_f16 = f16_out ? 1 : 0;
  if (planes_in) return pair ? launch<false, 2>(ma, mb, md, md, md, p, st) : launch<false, 1>(ma, mb, md, md, md, p, st);
  return pair ? launch<true, 2>(ma, mb, md, md, md, p, st) : launch<true, 1>(ma, mb, md, md, md, p, st);
}

cudaError_t launch_proj_tc(bool qkv, const void* x, const void* w, const float* bias, void* d0, void* d1, void* d2,
                           const jv_shape& s, int* status, cudaStream_t st) {
  if (!encode_fn()) return cudaErrorNotSupported;
  const uint64_t N = (uint64_t)shape_tokens(s), C = (uint64_t)s.H * kD, BH = (uint64_t)s.B * s.H;   // prefix and grid tokens alike
  const uint64_t features = qkv ? 3 * C : C;
  const bool pair = pair_tiles((int64_t)s.B * ceil_div((int)N, kBM), ceil_div((int)features, kBN));
  CUtensorMap ma, mb, md0, md1, md2;
  bool ok = map2(&mb, w, C, features, pair ? kBN / 2 : kBN);
  if (qkv) {
    ok = ok && map3(&ma, x, C, N, s.B, kBM) && map3(&md0, d0, kD, N, BH, 32) && map3(&md1, d1, kD, N, BH, 32) &&
         map3(&md2, d2, kD, N, BH, 32);
  } else {
    ok = ok && map3(&ma, x, kD, N, BH, kBM) && map3(&md0, d0, C, N, s.B, 32);
    md1 = md0;
    md2 = md0;
  }
  ProjParams p;
  if (!ok || !plan(p, pair, s.B, (int)N, (int)features, s.H, false)) return cudaErrorInvalidValue;
  p.bias = bias;
  p.bias_vec = ((uintptr_t)bias & 15) == 0;
  p.status = status;
  p.H = s.H;
  p.silu = 0;
  p.out_f16 = 0;
  if (qkv) return pair ? launch<true, 2>(ma, mb, md0, md1, md2, p, st) : launch<true, 1>(ma, mb, md0, md1, md2, p, st);
  return pair ? launch<false, 2>(ma, mb, md0, md1, md2, p, st) : launch<false, 1>(ma, mb, md0, md1, md2, p, st);
}

}  // namespace jv
