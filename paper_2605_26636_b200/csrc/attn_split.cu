// Full softmax attention (Eq. 1) one 128-row query tile at a time, its keys split over the four tile slots of a CTA: for problems
// of few query tiles, and for what whole rounds of the four-tile kernel (attn_f4.cu) leave over.  bf16 tensors, head_dim 64.
//
// What bounds such a call is the chain of one query tile: with a tile or two per CTA the steps of 64 keys follow each other
// through  scores -> softmax -> P V  at 0.7 us each, on SMs whose sub-cores hold one or two softmax warps.  Here the four slots
// hold the SAME queries and a quarter of the keys each, so a tile's chain is a quarter as long and every sub-core
// still has four softmax warps to overlap; the four partial softmaxes (row maximum, row sum, unnormalised output, all fp32)
// are merged through shared memory at the end.  A tile costs as much as a quarter of an item of four on the four-tile
// kernel, plus 4 us to fill the pipeline and to merge, and the work comes in four times finer pieces.
//
// Measured, before (the better of the four-tile and the two-tile kernel) / now, us: 6 heads of 1370 tokens 22.0 / 13.0, of 3038 tokens
// 44.3 / 22.3, of 5329 71 / 64; 24 of 576 13.3 / 8.9; 16 of 1030 20.7 / 12.3.  Behind whole rounds of four tiles: 12 heads of 6988 tokens
// 232 / 176, 64 of 5329 591 / 566 (in turn, in a loop at the power cap), 16 of 16384 1204 / 1152.
//
// Warp roles (19 warps): 0 TMA producer, 1 and 2 MMA issuers (slots 0, 1 and 2, 3), 3-18 softmax, one thread per query row
// and slot, then the merge, one thread per query row and 16 channels.  A slot has its own rings of K and V in boxes of 64 keys; when
// its last product has retired they take its partial output.  Tensor memory: per slot 64 columns of scores, with P
// over the first 32 of them, and 64 of output.
//
// Every mbarrier wait is bounded: a wait that runs out sets the device status word, raises a CTA-wide abort flag, and every
// role falls through to the common teardown (tensor memory is always released).
#include "tc_common.cuh"

namespace jv {
namespace {

using namespace tc;

constexpr uint32_t kSuspendNs = 4000;          // suspend-time hint of this kernel's barrier waits (tc_common.cuh)
constexpr int kD = 64;
constexpr int kTile = 128;                     // query rows
constexpr int kSub = 64;                       // keys per step
constexpr int kTileBytes = kTile * kD * 2;     // 16 KB
constexpr int kSubBytes = kSub * kD * 2;       // 8 KB
constexpr int kSlots = 4;
constexpr int kStages = 3;                     // depth of a slot's K ring and of its V ring, in boxes of 64 keys
constexpr int kSlotBytes = 2 * kStages * kSubBytes;
constexpr int kPartBytes = kTile * kD * 4;     // a slot's partial output, fp32: [channel / 4][row] 16-byte pieces
static_assert(kSlotBytes >= kPartBytes + kTile * 8, "partial output, then (maximum, sum) of every row");
constexpr int kWarps = 19;
constexpr int kThreads = kWarps * 32;
constexpr int kFirstSoftmaxWarp = 3;
constexpr uint32_t kTmemCols = 512;
constexpr int kPolyOf8 = 2;                    // of every 8 score pairs, this many take the polynomial exponential
constexpr uint32_t kColS = 0, kColO = 256;     // S_t (and P_t) at 64 t, O_t at 256 + 64 t
constexpr uint32_t kIdescQK = idesc(kTile, kSub, 0);
constexpr uint32_t kIdescPV = idesc(kTile, kD, 1);

struct SplitParams {
  __nv_bfloat16* o;
  int* status;
  int N;                  // tokens per (batch, head)
  int nbox;               // boxes of 64 keys per head
  int qgroups, rest;      // per head: whole groups of four query tiles, and tiles behind them
  int ragged;             // CTAs [0, ragged): the tiles behind the groups, head by head; then the tiles of the groups
  int first_group;        // from this one on (head by head; those before it are the four-tile kernel's)
  bool overlap;           // the launch ahead is that of the four-tile kernel on this call's other tiles
  FastDiv div_qgroups;
  int H;                  // heads per batch element: the inputs are addressed by (head, batch)
  FastDiv div_H;
  float scale_log2;       // softmax scale * log2(e)
};

struct __align__(8) Barriers {
  uint64_t q_full;
  uint64_t k_full[kSlots][kStages], k_empty[kSlots][kStages], v_full[kSlots][kStages], v_empty[kSlots][kStages];
  uint64_t s_full[kSlots], p_full[kSlots], o_full[kSlots];
  uint64_t drain;
  uint32_t tmem_base;
  volatile uint32_t abort_flag;
};
constexpr size_t kSmemTiles = kTileBytes + (size_t)kSlots * kSlotBytes;    // Q | per slot K[kStages] V[kStages]
constexpr size_t kSmemBytes = kSmemTiles + sizeof(Barriers) + 1024;        // + alignment slack
static_assert(kSmemBytes <= 232448, "shared memory of one CTA");

// boxes of slot s: [first_box(s), first_box(s + 1))
__device__ __forceinline__ int first_box(int s, int nbox) { return (s * nbox) / kSlots; }

__global__ void __launch_bounds__(kThreads, 1)
attn_split_kernel(const __grid_constant__ CUtensorMap mapQ, const __grid_constant__ CUtensorMap mapK,
                  const __grid_constant__ CUtensorMap mapV, const SplitParams p) {
  extern __shared__ unsigned char smem_raw[];
  if (threadIdx.x == 32) {
    prefetch_map(&mapQ);
    prefetch_map(&mapK);
    prefetch_map(&mapV);
  }
  // 1024-byte alignment by an offset from the array itself, so that accesses stay shared-space loads and stores
  unsigned char* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  Barriers* bar = reinterpret_cast<Barriers*>(smem + kSmemTiles);
  const uint32_t sQ = smem_u32(smem), sRing = sQ + kTileBytes;

  const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    mbar_init(&bar->q_full, 1);
    for (int t = 0; t < kSlots; ++t) {
      mbar_init(&bar->s_full[t], 1);
      mbar_init(&bar->p_full[t], 128);
      mbar_init(&bar->o_full[t], 1);
      for (int s = 0; s < kStages; ++s) {
        mbar_init(&bar->k_full[t][s], 1);
        mbar_init(&bar->k_empty[t][s], 1);
        mbar_init(&bar->v_full[t][s], 1);
        mbar_init(&bar->v_empty[t][s], 1);
      }
    }
    mbar_init(&bar->drain, 2);
    bar->abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 0) {
    __syncwarp();
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&bar->tmem_base)),
                 "r"(kTmemCols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = __shfl_sync(0xffffffffu, bar->tmem_base, 0);

  // What is read and written from here on may belong to the launch ahead; overlap: that launch has waited for what came
  // before it, and is waited for at the end.
  if (!p.overlap) griddep_wait();
  griddep_launch_dependents();
  // a timeout flagged earlier (by any CTA or launch) makes the rest leave at once
  if (threadIdx.x == 0 && *reinterpret_cast<volatile int*>(p.status) != 0) bar->abort_flag = 1;
  __syncthreads();
  if (bar->abort_flag) {
    if (warp == 0)
      asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
    if (p.overlap) griddep_wait();
    return;
  }

  int bh, qt;
  if ((int)blockIdx.x < p.ragged) {
    bh = blockIdx.x / p.rest;
    qt = 4 * p.qgroups + (blockIdx.x - bh * p.rest);
  } else {
    const int k = blockIdx.x - p.ragged, g = p.first_group + (k >> 2);
    bh = fdiv(g, p.div_qgroups);
    qt = 4 * (g - bh * p.qgroups) + (k & 3);
  }
  const int nbox = p.nbox;

  if (warp == 0) {
    // ================= TMA producer =================
    const int b = fdiv(bh, p.div_H), h = bh - b * p.H;   // coordinates of the input tensor maps
    if (elect_one()) {
      mbar_expect_tx(&bar->q_full, kTileBytes);
      tma_load_4d(sQ, &mapQ, &bar->q_full, 0, qt * kTile, h, b);
    }
    __syncwarp();
    bool ok = true;
    const int most = (nbox + kSlots - 1) / kSlots;       // steps of the longest slot
    int issued[kSlots] = {0, 0, 0, 0};                   // boxes whose copies are under way (for the abort path)
    for (int u = 0; u < most && ok; ++u) {
      const int st = u % kStages;
      const uint32_t par = ((u / kStages) & 1) ^ 1;
#pragma unroll
      for (int t = 0; t < kSlots; ++t) {
        const int box = first_box(t, nbox) + u;
        if (!ok || box >= first_box(t + 1, nbox)) continue;
        const uint32_t dk = sRing + t * kSlotBytes + st * kSubBytes, dv = dk + kStages * kSubBytes;
        ok = warp_wait<kSuspendNs>(&bar->k_empty[t][st], par, &bar->abort_flag, p.status);
        if (ok) ok = warp_wait<kSuspendNs>(&bar->v_empty[t][st], par, &bar->abort_flag, p.status);
        if (!ok) continue;
        if (elect_one()) {
          mbar_expect_tx(&bar->k_full[t][st], kSubBytes);
          tma_load_4d(dk, &mapK, &bar->k_full[t][st], 0, box * kSub, h, b);
          mbar_expect_tx(&bar->v_full[t][st], kSubBytes);
          tma_load_4d(dv, &mapV, &bar->v_full[t][st], 0, box * kSub, h, b);
        }
        __syncwarp();
        issued[t] = u + 1;
      }
    }
    if (!ok && lane == 0) {
      // let the copies still in flight land before the CTA leaves (bounded by the same limit)
      const unsigned long long t0 = globaltimer();
      while (!mbar_try(&bar->q_full, 0) && globaltimer() - t0 < kWaitLimitNs) {}
#pragma unroll
      for (int t = 0; t < kSlots; ++t)
        for (int g = max(0, issued[t] - kStages); g < issued[t]; ++g) {
          while (!mbar_try(&bar->k_full[t][g % kStages], (g / kStages) & 1) && globaltimer() - t0 < kWaitLimitNs) {}
          while (!mbar_try(&bar->v_full[t][g % kStages], (g / kStages) & 1) && globaltimer() - t0 < kWaitLimitNs) {}
        }
    }
  } else if (warp < kFirstSoftmaxWarp) {
    // ================= MMA issuers: warp 1 serves slots 0 and 1, warp 2 slots 2 and 3 =================
    // Per slot t a chain over its steps u:  O_t += P_t(u - 1) V(u - 1), then S_t(u) = Q K(u)^T.  P_t lies over S_t; one
    // thread's MMAs execute in issue order, so the commit that publishes S_t(u) also says that P_t(u - 1) V(u - 1) has retired.
    const int tb = 2 * (warp - 1);
    bool ok = warp_wait<kSuspendNs>(&bar->q_full, 0, &bar->abort_flag, p.status);
    const int n0 = first_box(tb + 1, nbox) - first_box(tb, nbox), n1 = first_box(tb + 2, nbox) - first_box(tb + 1, nbox);
    const int most = max(n0, n1);
    for (int u = 0; u <= most && ok; ++u) {
      const int sk = u % kStages, sv = (u + kStages - 1) % kStages;     // stages of K(u) and of V(u - 1)
      const uint32_t phk = (u / kStages) & 1, phv = u > 0 ? ((u - 1) / kStages) & 1 : 0;
#pragma unroll
      for (int x = 0; x < 2; ++x) {
        const int t = tb + x, n = x == 0 ? n0 : n1;
        if (!ok || u > n) continue;
        const bool has_qk = u < n, has_pv = u > 0;
        const uint32_t kb = sRing + t * kSlotBytes + sk * kSubBytes;
        const uint32_t vb = sRing + t * kSlotBytes + (kStages + sv) * kSubBytes;
        if (has_qk) ok = warp_wait<kSuspendNs>(&bar->k_full[t][sk], phk, &bar->abort_flag, p.status);
        if (ok && has_pv) {
          ok = warp_wait<kSuspendNs>(&bar->v_full[t][sv], phv, &bar->abort_flag, p.status);
          if (ok) ok = warp_wait<kSuspendNs>(&bar->p_full[t], (u - 1) & 1, &bar->abort_flag, p.status);
        }
        if (!ok) continue;
        tc_fence_after();
        if (elect_one()) {                 // one lane issues the step's MMAs back to back
          if (has_pv) {
            const uint64_t dv = smem_desc(vb);
#pragma unroll
            for (int ks = 0; ks < kSub / 16; ++ks)
              mma_ts_1(tmem + kColO + t * kD, tmem + kColS + t * kSub + ks * 8, desc_advance(dv, ks * 2048), kIdescPV,
                       (u > 1 || ks > 0) ? 1u : 0u);
          }
          if (has_qk) {
            const uint64_t dq = smem_desc(sQ), dk = smem_desc(kb);
#pragma unroll
            for (int ks = 0; ks < kD / 16; ++ks)
              mma_ss_1(tmem + kColS + t * kSub, desc_advance(dq, ks * 32), desc_advance(dk, ks * 32), kIdescQK, ks > 0);
          }
        }
        __syncwarp();
        if (has_qk) {
          tc_commit(&bar->s_full[t]);
          tc_commit(&bar->k_empty[t][sk]);
        } else {
          tc_commit(&bar->o_full[t]);
        }
        if (has_pv) tc_commit(&bar->v_empty[t][sv]);
      }
    }
    // Teardown: every MMA issued so far must have retired before tensor memory is released.
    tc_commit(&bar->drain);
    if (lane == 0) {
      const unsigned long long t0 = globaltimer();
      while (!mbar_try(&bar->drain, 0) && globaltimer() - t0 < kWaitLimitNs) {}
    }
    __syncwarp();
  } else {
    // ================= softmax: one thread per query row and slot =================
    const int t = (warp - kFirstSoftmaxWarp) >> 2;  // slot of this warp
    const int q4 = warp & 3;                        // tensor-memory quadrant a warp may touch: warp % 4
    const uint32_t lane_base = (uint32_t)(q4 << 5) << 16;
    const uint32_t tS = tmem + lane_base + kColS + t * kSub;   // scores; probabilities over their first 32 columns
    const uint32_t tO = tmem + lane_base + kColO + t * kD;
    const float sl2 = p.scale_log2;
    const float kLazy = 8.f / sl2;                 // the reference maximum moves only when it grew by > 2^8
    const uint64_t sl2x2 = pack2(sl2, sl2);
    const int box0 = first_box(t, nbox), nsteps = first_box(t + 1, nbox) - box0;
    const int last_valid = p.N - (nbox - 1) * kSub;            // keys that exist in the last box
    bool ok = true;
    float m = -INFINITY, l = 0.f;
    for (int u = 0; u < nsteps; ++u) {
      ok = warp_wait<kSuspendNs>(&bar->s_full[t], u & 1, &bar->abort_flag, p.status);
      if (!ok) break;
      tc_fence_after();
      uint32_t va[32];
      if (box0 + u == nbox - 1 && last_valid < kSub) {
        // the scores of keys that do not exist become -inf in tensor memory
#pragma unroll 1
        for (int c = 0; c < 2; ++c) {
          const int nv = last_valid - 32 * c;                    // valid keys among these 32
          if (nv < 32) {                                         // warp-uniform
            tmem_ld32(tS + 32 * c, va);
            tmem_wait_ld(va);
#pragma unroll
            for (int x = 0; x < 32; ++x)
              if (x >= nv) va[x] = kNegInf;
            tmem_st32(tS + 32 * c, va);
          }
        }
        tmem_wait_st();
      }
      // pass 1: the step's maximum (second half first, so that the first half is the one left in registers)
      float mx4[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
      tmem_ld32(tS + 32, va);
      tmem_wait_ld(va);
      max32(va, mx4);
      tmem_ld32(tS, va);
      tmem_wait_ld(va);
      max32(va, mx4);
      const float mx = max_of(mx4);
      float o_scale = 1.f;
      if (ref_moves(mx, m, kLazy)) { // always true on the first step, unless all of its scores are -inf
        o_scale = ref_scale(m, mx, sl2);
        l *= o_scale;
        m = mx;
      }
      if (u > 0 && __any_sync(0xffffffffu, o_scale != 1.f)) {
        // Rare: the reference moved.  O_t is quiescent: the scores just waited for were committed behind the previous step's P V.
#pragma unroll 1
        for (int c = 0; c < 2; ++c) {
          uint32_t v[32];
          tmem_ld32(tO + 32 * c, v);
          tmem_wait_ld(v);
#pragma unroll
          for (int x = 0; x < 32; ++x) v[x] = __float_as_uint(__uint_as_float(v[x]) * o_scale);
          tmem_st32(tO + 32 * c, v);
        }
        tmem_wait_st();
        tmem_ld32(tS, va);           // pass 2 needs the first half of the scores again
        tmem_wait_ld(va);
      }
      // pass 2: exponentials against the reference, P over the scores just consumed
      const float mneg = ref_negative(m, sl2);
      const uint64_t mnegx2 = pack2(mneg, mneg);
      uint64_t lsum[4] = {0ull, 0ull, 0ull, 0ull};
      uint32_t pk[16];
      exp32<false, kPolyOf8>(va, sl2x2, mnegx2, lsum, pk, mx4);
      tmem_st16(tS, pk);
      tmem_ld32(tS + 32, va);
      tmem_wait_ld(va);
      exp32<false, kPolyOf8>(va, sl2x2, mnegx2, lsum, pk, mx4);
      tmem_st16(tS + 16, pk);
      float a0, a1, b0, b1;
      unpack2(add2(lsum[0], lsum[1]), a0, a1);
      unpack2(add2(lsum[2], lsum[3]), b0, b1);
      l += (a0 + a1) + (b0 + b1);
      tmem_wait_st();
      tc_fence_before();
      mbar_arrive(&bar->p_full[t]);
    }
    if (ok) ok = warp_wait<kSuspendNs>(&bar->o_full[t], 0, &bar->abort_flag, p.status);
    if (ok) {
      // the slot's partial result over its own rings, which nothing reads any more
      tc_fence_after();
      const int row = 32 * q4 + lane;
      unsigned char* part = smem + kTileBytes + (size_t)t * kSlotBytes;
#pragma unroll 1
      for (int c = 0; c < 2; ++c) {
        uint32_t v[32];
        tmem_ld32(tO + 32 * c, v);
        tmem_wait_ld(v);
#pragma unroll
        for (int x = 0; x < 8; ++x)
          *reinterpret_cast<uint4*>(part + (size_t)((8 * c + x) * kTile + row) * 16) =
              make_uint4(v[4 * x], v[4 * x + 1], v[4 * x + 2], v[4 * x + 3]);
      }
      *reinterpret_cast<float2*>(part + kPartBytes + row * 8) = make_float2(m, l);
    }
  }

  __syncwarp();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp >= kFirstSoftmaxWarp && !bar->abort_flag) {
    // ================= merge: one thread per query row and 16 channels =================
    const int row = (threadIdx.x - 32 * kFirstSoftmaxWarp) & (kTile - 1), cq = (threadIdx.x - 32 * kFirstSoftmaxWarp) / kTile;
    const int tok = qt * kTile + row;
    const unsigned char* part = smem + kTileBytes;
    float2 ml[kSlots];
#pragma unroll
    for (int t = 0; t < kSlots; ++t) ml[t] = *reinterpret_cast<const float2*>(part + (size_t)t * kSlotBytes + kPartBytes + row * 8);
    const float M = fmaxf(fmaxf(ml[0].x, ml[1].x), fmaxf(ml[2].x, ml[3].x));
    float f[kSlots], L = 0.f;
#pragma unroll
    for (int t = 0; t < kSlots; ++t) {
      f[t] = ex2((ml[t].x - M) * p.scale_log2);
      L = fmaf(ml[t].y, f[t], L);
    }
    const float inv = 1.f / L;
    uint32_t out[8];
#pragma unroll
    for (int x = 0; x < 4; ++x) {
      float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int t = 0; t < kSlots; ++t) {
        const float4 y = *reinterpret_cast<const float4*>(part + (size_t)t * kSlotBytes + (size_t)((4 * cq + x) * kTile + row) * 16);
        a.x = fmaf(y.x, f[t], a.x);
        a.y = fmaf(y.y, f[t], a.y);
        a.z = fmaf(y.z, f[t], a.z);
        a.w = fmaf(y.w, f[t], a.w);
      }
      out[2 * x] = pack_bf16(a.x * inv, a.y * inv);
      out[2 * x + 1] = pack_bf16(a.z * inv, a.w * inv);
    }
    if (tok < p.N) {
      uint4* dst = reinterpret_cast<uint4*>(p.o + ((size_t)bh * p.N + tok) * kD + 16 * cq);
      dst[0] = make_uint4(out[0], out[1], out[2], out[3]);
      dst[1] = make_uint4(out[4], out[5], out[6], out[7]);
    }
  }
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
  if (p.overlap) griddep_wait();
}

// In steps of 64 keys of the four-tile kernel a round of tiles here takes a quarter of the steps of a head, and 3.5 more.  The
// comparison with the other kernels (2 steps of overhead) takes the faster side, or one within 2.5 % of it, over 6 to 192 heads of 320 to 8192
// tokens: 16 of 4096 101 us here / 86 there, 24 of 1024 20.2 / 18.0 (two tiles at a time), 64 of 4096 334 / 345, 48 of 2500 110.6 / 108.7.
// What of a call goes where: `groups` groups of four tiles to the four-tile kernel (whole rounds of it, or none), `tiles` here.
struct SplitPlan {
  int groups, tiles;
  float steps;            // time, in steps of 64 keys of the four-tile kernel
};
SplitPlan plan_split(int ntiles, int nbox, int BH) {
  const int sms = device_sm_count(), whole = ntiles / 4 * BH;
  SplitPlan best{0, 0, 0.f};
  for (int rounds = whole / sms; ; rounds = 0) {           // as many whole rounds as there are, or none
    const int tiles = ntiles * BH - 4 * sms * rounds;
    const float steps = rounds * (float)nbox + ceil_div(tiles, sms) * (0.25f * nbox + 3.5f);
    if (best.tiles == 0 || steps < best.steps) best = SplitPlan{rounds * sms, tiles, steps};
    if (rounds == 0) return best;
  }
}

}  // namespace

bool attn_split_supported(const AttnArgs& a) {
  if (a.dtype != JV_BF16 || a.D != kD) return false;
  const int64_t N = (int64_t)a.Hg * a.Wg;
  if (N <= 3 * kSub) return false;                       // every slot needs a box of its own
  const int64_t ntiles = (N + kTile - 1) / kTile, nbox = (N + kSub - 1) / kSub;
  if (ntiles * a.BH > 0x7fffffffll) return false;
  if (plan_split((int)ntiles, (int)nbox, a.BH).steps > attn_f4_cost((int)ntiles, a.BH) * nbox + 2.f) return false;
  return encode_fn() != nullptr;
}

cudaError_t launch_attn_split(const AttnArgs& a, int* status, cudaStream_t st) {
  EncodeFn enc = encode_fn();
  if (!enc) return cudaErrorNotSupported;
  const int N = a.Hg * a.Wg;
  CUtensorMap maps[3];
  const void* ptrs[3] = {a.q, a.k, a.v};
  // the inputs as (d, token, head, batch) with the caller's strides
  const cuuint64_t dims[4] = {(cuuint64_t)kD, (cuuint64_t)N, (cuuint64_t)a.H, (cuuint64_t)(a.BH / a.H)};
  const cuuint64_t strides[3] = {(cuuint64_t)a.in.tok * 2, (cuuint64_t)a.in.head * 2, (cuuint64_t)a.in.batch * 2};
  const cuuint32_t estr[4] = {1, 1, 1, 1};
  for (int i = 0; i < 3; ++i) {
    const cuuint32_t box[4] = {(cuuint32_t)kD, (cuuint32_t)(i == 0 ? kTile : kSub), 1, 1};
    if (enc(&maps[i], CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(ptrs[i]), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
      return cudaErrorInvalidValue;
  }
  static OncePerDevice smem_opt_in;   // > 48 KB of dynamic shared memory: a per-device function attribute
  const cudaError_t e = smem_opt_in.run(
      [] { return cudaFuncSetAttribute(attn_split_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemBytes); });
  if (e != cudaSuccess) return e;
  SplitParams p;
  p.o = (__nv_bfloat16*)a.o;
  p.status = status;
  p.N = N;
  p.nbox = ceil_div(N, kSub);
  const int ntiles = ceil_div(N, kTile);
  const SplitPlan plan = plan_split(ntiles, p.nbox, a.BH);
  p.qgroups = ntiles / 4;
  p.rest = ntiles % 4;
  p.ragged = p.rest * a.BH;
  p.first_group = plan.groups;
  p.overlap = plan.groups > 0;
  p.div_qgroups = make_fastdiv((uint32_t)(p.qgroups > 0 ? p.qgroups : 1));
  p.H = a.H;
  p.div_H = make_fastdiv((uint32_t)a.H);
  p.scale_log2 = a.scale * 1.4426950408889634f;
  if (plan.groups > 0) {
    const cudaError_t f = launch_attn_f4(a, status, st, plan.groups);
    if (f != cudaSuccess) return f;
  }
  return launch_programmatic(attn_split_kernel, dim3(plan.tiles), kThreads, kSmemBytes, st, maps[0], maps[1], maps[2], p);
}

}  // namespace jv
