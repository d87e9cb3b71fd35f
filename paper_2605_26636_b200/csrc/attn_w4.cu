// 2-D window attention (Sec. 3.2.2) for windows of one or two 128-token tiles (16 x 16 and the like) and of 8 x 8
// tokens on the 5th-generation tensor cores: two windows (pairs, fours of small ones) side by side per CTA, four 128-row
// query tiles, so that every SM sub-core holds four softmax warps.  bf16 tensors, head_dim 64, at most 16 prefix tokens.
//
// The softmax of attention at head_dim 64 is bound by the SM's ordinary pipes and their latencies, and a
// window is short work (four 64-key steps per query tile): with two query tiles per CTA (attn_tc.cu) a
// sub-core has two warps to overlap a step's chain  scores -> softmax -> P V  with.  Here a CTA is
// two independent halves ("slots"); each slot walks its own sequence of items with its own producer
// warp, issuer warp, eight softmax warps and rings of K and V, and shares nothing with the other
// but the SM.  The two slots drift out of phase, so one slot's epilogue and pipeline fill overlap the
// other's steady state.
//
// An item is up to two query tiles, one above the other (template parameter kWpt, windows per tile):
//   kWpt = 0   one window of up to two tiles: both query tiles attend all its keys
//   kWpt = 1   two windows of one tile each: a query tile attends its own keys only
//   kWpt = 2   four windows of 8 x 8 tokens: a tile is two of them side by side, a row attends the 64 of its tile's
//              128 keys that lie in its own half (of every 16 columns of the scores, 8 belong to the row: they are
//              selected in registers, only they get an exponential, and P is zero elsewhere)
//
// Warp roles (20 warps):
//   warps 0, 1    TMA producers of slot 0 / 1: per item two Q tiles (each double-buffered: the next item's Q is on its
//                 way while this one is worked on), K and V in boxes of 64 keys through rings
//   warps 2, 3    MMA issuers of slot 0 / 1, in steps of 64 keys, both query tiles of the item:
//                 O_t += P_t V (A = P from tensor memory) of the previous step, then S_t = Q_t K^T
//   warps 4-19    softmax, one thread per query row (warp w: tile (w - 4) / 4, tensor-memory quadrant w % 4):
//                 exact two-pass softmax per step against a lazily raised reference, P as bf16 over
//                 the scores it came from, final 1/l scaling, store
// Tensor memory: per tile a 64-column score buffer and a 64-column accumulator (4 x 128 = 512 columns).
// Shared memory (224 KB): Q 8 tiles, per slot a K ring of two boxes and a V ring of four (three with prefix tokens, whose
// rows of K and V, one more step per window, take the room).  The output tile is staged over its own Q tile; the
// producer may refill that buffer when the four warps that staged into it have seen their stores read it, which they
// check one step into their next item, off the critical path.
//
// Measured (8 x 16 heads, 64 x 64 tokens, 16 x 16 windows): 55 us = 4.85 TB/s in short runs, 65.5 in a long loop at the power cap; with five
// prefix tokens (their queries' kernel, 29 us, included) 89 and 100.  With one Q buffer per tile, K and V in whole tiles and the output staged over
// V it was 60 and 71 (114 and 119): a window's Q could only be copied once the window before had issued its last scores, and there was no
// room for a third V stage beside the prefix rows.  8 x 8 windows, 32 x 12 heads of 16 x 16 tokens 12.8 us, 8 x 16 of 64 x 64 46.1 (on attn_tc.cu, where
// half of a tile's rows, and half of the exponentials of the rest, are of no use, 186).
//
// Every mbarrier wait is bounded: a wait that runs out sets the device status word, raises a
// CTA-wide abort flag, and every role falls through to the common teardown (tensor memory is
// always released).
#include "tc_common.cuh"

namespace jv {
namespace {

using namespace tc;

#ifndef JV_ATTN_SUSPEND_NS
#define JV_ATTN_SUSPEND_NS 4000
#endif
constexpr uint32_t kSuspendNs = JV_ATTN_SUSPEND_NS;   // suspend-time hint of this kernel's barrier waits (tc_common.cuh)
constexpr int kD = 64;
constexpr int kTile = 128;                  // tokens per tile (MMA M and key-tile rows)
constexpr int kTileBytes = kTile * kD * 2;  // 16 KB
constexpr int kSlots = 2;                   // windows in flight per CTA
constexpr int kQT = 2 * kSlots;             // query tiles per CTA
constexpr int kKS = 2;                      // K ring depth per slot, in boxes of 64 keys
constexpr int kVSMax = 4;                   // V ring depth per slot: 4 boxes without prefix tokens, 3 with them
constexpr int kPreRows = 16;                // prefix keys are one 16-key MMA: P <= 16
constexpr int kPreBytes = kPreRows * kD * 2;   // 2 KB: the prefix rows of K, or of V
constexpr int kWarps = 20;
constexpr int kThreads = kWarps * 32;
constexpr int kFirstSoftmaxWarp = 4;
constexpr uint32_t kTmemCols = 512;
constexpr int kSub = 64;                    // keys per step
constexpr int kSubBytes = kSub * kD * 2;    // 8 KB
constexpr int kPolyOf8 = 2;                 // of every 8 score pairs, this many take the polynomial exponential
// Tensor-memory columns: S_t (and P_t over its first 32 columns) at 64 t, O_t at 256 + 64 t
constexpr uint32_t kColS = 0, kColO = 256;

struct W4Params {
  int P;                 // prefix keys behind every window's own keys (0: none)
  int* status;
  int gridW, gridH;      // token grid
  int win_w, win_h;      // extent of an item: win_w == box_w, win_h == box_h or 2 * box_h
  int box_w, box_h;      // tile box: box_w * box_h == 128
  int lg_box_w;
  int nwx, nwin;         // items per grid row, per (batch, head)
  int total;             // items of the whole call: (batch*head, item), item fastest
  FastDiv div_nwin, div_nwx;
  int H;                 // heads per batch element: the inputs are addressed by (head, batch)
  FastDiv div_H;
  float scale_log2;      // softmax scale * log2(e)
};

// One item of one (batch, head)
struct Item {
  int bh, x0, y0, x_end, y_end;   // origin and valid end (exclusive) in the token grid
  int ntiles;                     // query tiles (1 or 2)
  int nsteps;                     // steps of 64 keys against the item's own keys
};
template <int kWpt>
__device__ __forceinline__ Item decode_item(const W4Params& p, int r) {
  Item it;
  it.bh = fdiv(r, p.div_nwin);
  const int win = r - it.bh * p.nwin;
  const int wy = fdiv(win, p.div_nwx), wx = win - wy * p.nwx;
  it.x0 = wx * p.win_w;
  it.y0 = wy * p.win_h;
  it.x_end = min(it.x0 + p.win_w, p.gridW);
  it.y_end = min(it.y0 + p.win_h, p.gridH);
  const int vh = it.y_end - it.y0, lg_half = 6 - p.lg_box_w;   // a step is 64 / box_w rows of the box
  it.ntiles = vh > p.box_h ? 2 : 1;
  it.nsteps = (vh + (1 << lg_half) - 1) >> lg_half;            // no step for rows that do not exist
  if (kWpt > 0) it.nsteps = min(it.nsteps, 2);
  return it;
}

struct __align__(8) Barriers {
  uint64_t q_full[kQT][2], q_empty[kQT][2];
  uint64_t k_full[kSlots][kKS], k_empty[kSlots][kKS], v_full[kSlots][kVSMax], v_empty[kSlots][kVSMax];
  uint64_t pre_full[kSlots], pre_empty[kSlots];       // the slot's prefix rows of K and V
  uint64_t s_full[kQT], p_full[kQT], o_full[kQT];
  uint64_t drain;
  uint32_t tmem_base;
  volatile uint32_t abort_flag;
};
// shared memory: Q[4][2] | K[2][kKS] | V[2][kVS] | (prefix variant: per slot the prefix rows of K, then of V) | barriers
template <bool kPrefix>
struct Layout {
  static constexpr int kVS = kPrefix ? 3 : 4;
  static constexpr size_t kTiles = (size_t)kQT * 2 * kTileBytes + (size_t)kSlots * (kKS + kVS) * kSubBytes;
  static constexpr size_t kPre = kPrefix ? (size_t)kSlots * 2 * kPreBytes : 0;
  static constexpr size_t kBytes = kTiles + kPre + sizeof(Barriers) + 1024;          // + alignment slack
  static_assert(kBytes <= 232448, "shared memory of one CTA");
};

constexpr uint32_t kIdescQK = idesc(kTile, kSub, 0);
constexpr uint32_t kIdescPV = idesc(kTile, kD, 1);
constexpr uint32_t kIdescQKpre = idesc(kTile, kPreRows, 0);   // scores against the 16 prefix rows

__device__ __forceinline__ void tma_store_4d(const CUtensorMap* map, uint32_t src, int c0, int c1, int c2, int c3) {
  asm volatile("cp.async.bulk.tensor.4d.global.shared::cta.tile.bulk_group [%0, {%2, %3, %4, %5}], [%1];"
               ::"l"(map), "r"(src), "r"(c0), "r"(c1), "r"(c2), "r"(c3) : "memory");
}

// ---- the kernel ------------------------------------------------------------------
// Slot s of CTA c works on items c + s * gridDim.x, then every 2 * gridDim.x-th.  Every role of a slot walks that
// sequence on its own; ring stages and barrier parities follow running counters.  The second query
// tile of an item that has one tile only (a bottom edge) is skipped by its softmax warps.
// kPrefix: every window's queries also attend the P <= 16 prefix tokens of their (batch, head): one more
// step per window with a 16-key score MMA against the prefix rows of K (kept in shared memory per slot,
// reloaded per window from L2) and a 16-key P V.  The prefix QUERIES are not this kernel's work.
template <bool kPrefix, int kWpt>
__global__ void __launch_bounds__(kThreads, 1)
attn_w4_kernel(const __grid_constant__ CUtensorMap mapQ, const __grid_constant__ CUtensorMap mapK,
               const __grid_constant__ CUtensorMap mapV, const __grid_constant__ CUtensorMap mapO,
               const __grid_constant__ CUtensorMap mapKp, const __grid_constant__ CUtensorMap mapVp, const W4Params p) {
  constexpr int kVS = Layout<kPrefix>::kVS;
  constexpr size_t kSmemTiles = Layout<kPrefix>::kTiles;
  extern __shared__ unsigned char smem_raw[];
  if (threadIdx.x == 32) {
    prefetch_map(&mapQ);
    prefetch_map(&mapK);
    prefetch_map(&mapV);
    prefetch_map(&mapO);
  }
  // 1024-byte alignment by an offset from the array itself, so that accesses stay shared-space loads and stores
  unsigned char* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  Barriers* bar = reinterpret_cast<Barriers*>(smem + kSmemTiles + Layout<kPrefix>::kPre);
  const uint32_t sQ = smem_u32(smem), sK = sQ + kQT * 2 * kTileBytes, sV = sK + kSlots * kKS * kSubBytes;
  const uint32_t sPre = sQ + (uint32_t)kSmemTiles;   // slot s: prefix rows of K at s * 4 KB, of V 2 KB behind them

  const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    for (int t = 0; t < kQT; ++t) {
      for (int b = 0; b < 2; ++b) {
        mbar_init(&bar->q_full[t][b], 1);
        mbar_init(&bar->q_empty[t][b], 4);   // handed back by the four softmax warps that staged their output into it
      }
      mbar_init(&bar->s_full[t], 1);
      mbar_init(&bar->p_full[t], 128);
      mbar_init(&bar->o_full[t], 1);
    }
    for (int s = 0; s < kSlots; ++s) {
      for (int g = 0; g < kKS; ++g) {
        mbar_init(&bar->k_full[s][g], 1);
        mbar_init(&bar->k_empty[s][g], 1);
      }
      for (int g = 0; g < kVS; ++g) {
        mbar_init(&bar->v_full[s][g], 1);
        mbar_init(&bar->v_empty[s][g], 1);
      }
      mbar_init(&bar->pre_full[s], 1);
      mbar_init(&bar->pre_empty[s], 1);
    }
    mbar_init(&bar->drain, kSlots);
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

  // With prefix tokens the launch ahead is that of their queries, which this one overlaps (it has waited for what came before
  // it before it let this one go); this one waits for it at its end.
  if (!kPrefix) griddep_wait();   // what is read and written from here on may belong to the launch ahead
  griddep_launch_dependents();
  // a timeout flagged earlier (by any CTA or launch) makes the rest leave at once
  if (threadIdx.x == 0 && *reinterpret_cast<volatile int*>(p.status) != 0) bar->abort_flag = 1;
  __syncthreads();
  if (bar->abort_flag) {
    if (warp == 0)
      asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
    if (kPrefix) griddep_wait();    // (no launch ends before the one ahead of it)
    return;
  }

  const int item_step = kSlots * gridDim.x;

  if (warp < kSlots) {
    // ================= TMA producer of slot `warp` =================
    const int s = warp;
    bool ok = true;
    int n = 0;                       // items seen
    int nq[2] = {0, 0};              // Q tiles issued per query tile
    int ks = 0, vs = 0;              // ring stages of the next K and V box
    uint32_t kpar = 1, vpar = 1;     // parity of the "empty" phase this pass over each ring waits for
    int issued_v = 0;                // for the abort path: V copies issued so far
    for (int r = blockIdx.x + s * gridDim.x; r < p.total && ok; r += item_step) {
      const Item it = decode_item<kWpt>(p, r);
      const int b = fdiv(it.bh, p.div_H), h = it.bh - b * p.H;   // coordinates of the input tensor maps
      const int half_h = p.box_h >> 1;
#pragma unroll
      for (int x = 0; x < 2; ++x) {
        if (x >= it.ntiles || !ok) continue;
        const int t = 2 * s + x, qb = nq[x] & 1;
        ok = warp_wait<kSuspendNs>(&bar->q_empty[t][qb], ((nq[x] >> 1) & 1) ^ 1, &bar->abort_flag, p.status);
        if (!ok) continue;
        if (elect_one()) {
          mbar_expect_tx(&bar->q_full[t][qb], kTileBytes);
          tma_load_5d(sQ + (2 * t + qb) * kTileBytes, &mapQ, &bar->q_full[t][qb], 0, it.x0, it.y0 + x * p.box_h, h, b);
        }
        __syncwarp();
        ++nq[x];
      }
      const int per_step = kWpt == 0 ? 1 : it.ntiles;  // key boxes per step: shared by the query tiles, or one each
      for (int u = 0; u < it.nsteps && ok; ++u) {      // in the order the issuer needs them: K of a step, V of it
        for (int x = 0; x < per_step && ok; ++x) {
          ok = warp_wait<kSuspendNs>(&bar->k_empty[s][ks], kpar, &bar->abort_flag, p.status);
          if (!ok) break;
          if (elect_one()) {
            mbar_expect_tx(&bar->k_full[s][ks], kSubBytes);
            tma_load_5d(sK + (s * kKS + ks) * kSubBytes, &mapK, &bar->k_full[s][ks], 0, it.x0, it.y0 + x * p.box_h + u * half_h, h, b);
          }
          __syncwarp();
          if (++ks == kKS) { ks = 0; kpar ^= 1; }
        }
        for (int x = 0; x < per_step && ok; ++x) {
          ok = warp_wait<kSuspendNs>(&bar->v_empty[s][vs], vpar, &bar->abort_flag, p.status);
          if (!ok) break;
          if (elect_one()) {
            mbar_expect_tx(&bar->v_full[s][vs], kSubBytes);
            tma_load_5d(sV + (s * kVS + vs) * kSubBytes, &mapV, &bar->v_full[s][vs], 0, it.x0, it.y0 + x * p.box_h + u * half_h, h, b);
          }
          __syncwarp();
          ++issued_v;
          if (++vs == kVS) { vs = 0; vpar ^= 1; }
        }
      }
      if (kPrefix && ok) {            // the prefix rows of K and V of this (batch, head): rows past P arrive as zeros
        ok = warp_wait<kSuspendNs>(&bar->pre_empty[s], (n & 1) ^ 1, &bar->abort_flag, p.status);
        if (!ok) break;
        if (elect_one()) {
          mbar_expect_tx(&bar->pre_full[s], 2 * kPreBytes);
          tma_load_4d(sPre + s * 2 * kPreBytes, &mapKp, &bar->pre_full[s], 0, 0, h, b);
          tma_load_4d(sPre + s * 2 * kPreBytes + kPreBytes, &mapVp, &bar->pre_full[s], 0, 0, h, b);
        }
        __syncwarp();
      }
      ++n;
    }
    if (!ok && lane == 0) {
      // let the copies still in flight land before the CTA leaves (bounded by the same limit): those of V by their
      // barriers, those of K and Q around them by a millisecond from here
      const unsigned long long t0 = globaltimer();
      for (int g = max(0, issued_v - kVS); g < issued_v; ++g)
        while (!mbar_try(&bar->v_full[s][g % kVS], (g / kVS) & 1) && globaltimer() - t0 < kWaitLimitNs) {}
      while (globaltimer() - t0 < 1000000ull) {}
    }
  } else if (warp < 2 * kSlots) {
    // ================= MMA issuer of slot `warp - 2`: both query tiles of the slot's item =================
    // Per item and query tile t the work is a chain over 64-key steps u:
    //   S_t(u) = Q_t K(u)^T          4 MMAs, M128 N64 K16, operands in shared memory
    //   O_t   += P_t(u) V(u)         4 MMAs, M128 N64 K16, A = P in tensor memory
    // P_t(u) lies over S_t(u), so S_t(u + 1) is issued behind P_t(u) V(u): the tensor pipe executes one
    // thread's MMAs in issue order.  The commit that publishes S_t(u + 1) therefore also tells the
    // softmax warps that P_t(u) V(u) has retired and O_t is quiescent.
    const int s = warp - kSlots, tb = 2 * s;
    bool ok = true;
    int sk = 0, sv = 0;                     // ring stages of the step's first score keys and P V keys
    uint32_t phk = 0, phv = 0;              // and their "full" parities
    uint32_t pcnt[2] = {0, 0};              // steps published so far per tile: parity of p_full
    uint32_t qcnt[2] = {0, 0};              // items in which the tile existed: buffer and parity of q_full
    uint32_t pre_cnt = 0;                   // items seen: parity of pre_full
    for (int r = blockIdx.x + s * gridDim.x; r < p.total && ok; r += item_step) {
      const Item it = decode_item<kWpt>(p, r);
      const int nsteps = it.nsteps;                   // steps against the item's own keys
      const int ns = nsteps + (kPrefix ? 1 : 0);      // and, behind them, one against the prefix rows
      const int per_step = kWpt == 0 ? 1 : it.ntiles; // key boxes per step
      for (int u = 0; u <= ns && ok; ++u) {
        const bool has_qk = u < nsteps, has_pre_qk = kPrefix && u == nsteps;          // scores of step u
        const bool has_pv = u > 0 && u <= nsteps, has_pre_pv = kPrefix && u == ns;    // P V of step u - 1
        if (has_pre_qk) {                   // the prefix rows of K and V must have landed
          ok = warp_wait<kSuspendNs>(&bar->pre_full[s], pre_cnt & 1, &bar->abort_flag, p.status);
          ++pre_cnt;
          if (!ok) break;
        }
        const uint32_t kpb = sPre + s * 2 * kPreBytes, vpb = kpb + kPreBytes;
        uint32_t kb = 0, vb = 0;
#pragma unroll
        for (int x = 0; x < 2; ++x) {
          if (x >= it.ntiles) continue;
          const int t = tb + x;
          if (has_qk && (x == 0 || kWpt > 0)) {        // a new key box: its K must have landed
            const int g = sk + x < kKS ? sk + x : sk + x - kKS;
            ok = warp_wait<kSuspendNs>(&bar->k_full[s][g], phk ^ (sk + x >= kKS), &bar->abort_flag, p.status);
            if (!ok) break;
            kb = sK + (s * kKS + g) * kSubBytes;
          }
          if (has_pv && (x == 0 || kWpt > 0)) {        // and the V of the step before
            const int g = sv + x < kVS ? sv + x : sv + x - kVS;
            ok = warp_wait<kSuspendNs>(&bar->v_full[s][g], phv ^ (sv + x >= kVS), &bar->abort_flag, p.status);
            if (!ok) break;
            vb = sV + (s * kVS + g) * kSubBytes;
          }
          const uint32_t qb = sQ + (2 * t + (qcnt[x] & 1)) * kTileBytes;
          if (u == 0) {
            ok = warp_wait<kSuspendNs>(&bar->q_full[t][qcnt[x] & 1], (qcnt[x] >> 1) & 1, &bar->abort_flag, p.status);
          } else {
            ok = warp_wait<kSuspendNs>(&bar->p_full[t], pcnt[x] & 1, &bar->abort_flag, p.status);
            ++pcnt[x];
          }
          if (!ok) break;
          tc_fence_after();
          if (elect_one()) {                 // one lane issues the step's MMAs back to back
            if (has_pv) {
              const uint64_t dv = smem_desc(vb);
#pragma unroll
              for (int c = 0; c < kSub / 16; ++c)
                mma_ts_1(tmem + kColO + t * kD, tmem + kColS + t * kSub + c * 8, desc_advance(dv, c * 2048), kIdescPV,
                         (u > 1 || c > 0) ? 1u : 0u);
            }
            if (has_pre_pv)                  // 16 prefix keys: one MMA of K = 16
              mma_ts_1(tmem + kColO + t * kD, tmem + kColS + t * kSub, smem_desc(vpb), kIdescPV, 1u);
            if (has_qk) {
              const uint64_t dq = smem_desc(qb), dk = smem_desc(kb);
#pragma unroll
              for (int c = 0; c < kD / 16; ++c)
                mma_ss_1(tmem + kColS + t * kSub, desc_advance(dq, c * 32), desc_advance(dk, c * 32), kIdescQK, c > 0);
            }
            if (has_pre_qk) {                // scores against the prefix rows: 16 columns
              const uint64_t dq = smem_desc(qb), dk = smem_desc(kpb);
#pragma unroll
              for (int c = 0; c < kD / 16; ++c)
                mma_ss_1(tmem + kColS + t * kSub, desc_advance(dq, c * 32), desc_advance(dk, c * 32), kIdescQKpre, c > 0);
            }
          }
          __syncwarp();
          if (u < ns) tc_commit(&bar->s_full[t]);
          else {
            tc_commit(&bar->o_full[t]);
            ++qcnt[x];
          }
        }
        if (!ok) break;
        for (int x = 0; x < per_step; ++x) {
          if (has_pv) {
            tc_commit(&bar->v_empty[s][sv]);
            if (++sv == kVS) { sv = 0; phv ^= 1; }
          }
          if (has_qk) {
            tc_commit(&bar->k_empty[s][sk]);
            if (++sk == kKS) { sk = 0; phk ^= 1; }
          }
        }
        if (has_pre_pv) tc_commit(&bar->pre_empty[s]);
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
    // ================= softmax + epilogue: one thread per query row =================
    const int t = (warp - kFirstSoftmaxWarp) >> 2;  // query tile of this warp
    const int s = t >> 1, x = t & 1;                // its slot, and which of the window's two tiles
    const int q4 = warp & 3;                        // tensor-memory quadrant a warp may touch: warp % 4
    const uint32_t lane_base = (uint32_t)(q4 << 5) << 16;
    const uint32_t tS = tmem + lane_base + kColS + t * kSub;   // scores; probabilities over their first 32 columns
    const uint32_t tO = tmem + lane_base + kColO + t * kD;
    const float sl2 = p.scale_log2;
    // The reference maximum moves only when it grew by > 2^8.  kWpt == 2: whenever it grew.  A window of 64 keys may have one that outweighs
    // all others; against the window's own maximum its probability is 1, which rounding to bf16 leaves alone (against that of the first half
    // of the keys: error 2.20e-3 of the result's norm, not 2.11e-3).
    const float kLazy = kWpt == 2 ? 0.f : 8.f / sl2;
    const uint64_t sl2x2 = pack2(sl2, sl2);
    const int sub_y = q4 * (p.box_h >> 2);          // this warp's 32 rows are box_h / 4 whole box rows
    bool ok = true;
    uint32_t scnt = 0;                // steps seen by this tile: parity of s_full
    uint32_t n = 0;                   // items in which this tile existed: buffer of its Q tile, parity of o_full
    int held = -1;                    // Q buffer this warp staged its last output into and has not handed back yet

    // hand back the buffer once this warp's store has read it (nothing to wait for if the warp stored nothing)
    auto release = [&]() {
      if (held >= 0) {
        if (lane == 0) {
          asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
          mbar_arrive(&bar->q_empty[t][held]);
        }
        __syncwarp();
        held = -1;
      }
    };

    for (int r = blockIdx.x + s * gridDim.x; r < p.total && ok; r += item_step) {
      const Item it = decode_item<kWpt>(p, r);
      if (x >= it.ntiles) continue;                   // this query tile does not exist
      const int nsteps = it.nsteps;                   // steps against the item's own keys
      const int ns = nsteps + (kPrefix ? 1 : 0);      // and, behind them, one against the prefix rows
      const int vx = it.x_end - it.x0;                // valid columns of every box of this item
      const int half_h = p.box_h >> 1;
      float m = -INFINITY, l = 0.f;
      for (int u = 0; u < ns; ++u) {
        const bool pre = kPrefix && u == nsteps;      // the step of the prefix keys: 16 score columns, P of them keys
        ok = warp_wait<kSuspendNs>(&bar->s_full[t], scnt & 1, &bar->abort_flag, p.status);
        if (!ok) break;
        ++scnt;
        tc_fence_after();
        uint32_t va[32];
        const int vy = it.y_end - (it.y0 + (kWpt == 0 ? 0 : x * p.box_h) + u * half_h);   // valid rows of this step's box
        const bool edge = vx < p.box_w || vy < half_h;
        // kWpt == 2: the row's own 32 of the step's 64 scores, -inf where the key does not exist
        auto load_own = [&]() {
          uint32_t vb[32];
          tmem_ld32(tS, va);
          tmem_ld32(tS + 32, vb);
          tmem_wait_ld(va);
          tmem_wait_ld(vb);
          const bool right = (lane >> 3) & 1;          // which of the tile's two windows this row belongs to
#pragma unroll
          for (int g = 0; g < 4; ++g)
#pragma unroll
            for (int i = 0; i < 8; ++i) {
              const uint32_t a = g < 2 ? va[16 * g + i] : vb[16 * (g - 2) + i];
              const uint32_t b = g < 2 ? va[16 * g + 8 + i] : vb[16 * (g - 2) + 8 + i];
              // in place: entry 8 g + i is read by this row of the loop only for g = 0 and never after it is written
              const uint32_t w = right ? b : a;
              if (g < 2) va[8 * g + i] = w;
              else vb[8 * (g - 2) + i] = w;
            }
#pragma unroll
          for (int i = 0; i < 16; ++i) va[16 + i] = vb[i];
          if (edge) {
            const int nv = vx - (right ? 8 : 0);       // valid columns of this row's window
#pragma unroll
            for (int i = 0; i < 32; ++i)
              if ((i & 7) >= nv || (i >> 3) >= vy) va[i] = kNegInf;
          }
        };
        if (pre) {
          // Columns 0 .. P - 1 hold the scores against the prefix keys; up to column 31 everything else
          // (scores against the zero rows behind them, the previous step's leftovers) becomes -inf.
          tmem_ld32(tS, va);
          tmem_wait_ld(va);
#pragma unroll
          for (int i = 0; i < 32; ++i)
            if (i >= p.P) va[i] = kNegInf;
          tmem_st32(tS, va);
          tmem_wait_st();
        } else if (kWpt != 2 && edge) {
          // Edge box: overwrite the scores of keys outside the grid with -inf in tensor memory, then
          // treat the step like any other.
#pragma unroll 1
          for (int c = 0; c < 2; ++c) {
            const int k0 = 32 * c;                     // first of the 32 keys, as an index into the box
            uint32_t bits = 0;
            if (p.box_w >= 32) {                       // the 32 keys lie in one box row
              const int ly = k0 >> p.lg_box_w, lx0 = k0 & (p.box_w - 1);
              const int nv = min(32, vx - lx0);
              if (ly < vy && nv > 0) bits = nv >= 32 ? 0xffffffffu : ((1u << nv) - 1u);
            } else {                                   // 32 / box_w whole box rows
              const uint32_t rowbits = (1u << min(vx, p.box_w)) - 1u;
              const int ly0 = k0 >> p.lg_box_w;
              for (int rr = 0; rr < (32 >> p.lg_box_w); ++rr)
                if (ly0 + rr < vy) bits |= rowbits << (rr << p.lg_box_w);
            }
            if (bits != 0xffffffffu) {                 // warp-uniform: the mask depends on the box only
              tmem_ld32(tS + 32 * c, va);
              tmem_wait_ld(va);
#pragma unroll
              for (int i = 0; i < 32; ++i)
                if (!((bits >> i) & 1u)) va[i] = kNegInf;   // exp2(-inf) = 0 and -inf never wins the maximum
              tmem_st32(tS + 32 * c, va);
            }
          }
          tmem_wait_st();
        }
        // ---- pass 1: the step's maximum (second half first, so that the first half is the one
        // left in registers for pass 2)
        float mx4[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
        if (kWpt == 2 && !pre) {
          load_own();
        } else {
          if (!pre) {
            tmem_ld32(tS + 32, va);
            tmem_wait_ld(va);
            max32(va, mx4);
          }
          tmem_ld32(tS, va);
          tmem_wait_ld(va);
        }
        max32(va, mx4);
        const float mx = max_of(mx4);
        float o_scale = 1.f;
        if (ref_moves(mx, m, kLazy)) { // always true on the first step, unless all of its scores are -inf
          o_scale = ref_scale(m, mx, sl2);            // first step: 0
          l *= o_scale;
          m = mx;
        }
        if (u > 0 && __any_sync(0xffffffffu, o_scale != 1.f)) {
          // The reference moved (rare, but for kWpt == 2).  O_t may be touched: the scores just waited for were committed
          // behind the previous step's P V, and the next P V waits for this step's P.
#pragma unroll 1
          for (int c = 0; c < 2; ++c) {
            uint32_t v[32];
            tmem_ld32(tO + 32 * c, v);
            tmem_wait_ld(v);
#pragma unroll
            for (int i = 0; i < 32; ++i) v[i] = __float_as_uint(__uint_as_float(v[i]) * o_scale);
            tmem_st32(tO + 32 * c, v);
          }
          tmem_wait_st();
          if (kWpt != 2) {                             // pass 2 needs the first half of the scores again
            tmem_ld32(tS, va);
            tmem_wait_ld(va);
          } else if (pre) {
            tmem_ld32(tS, va);
            tmem_wait_ld(va);
          } else {
            load_own();
          }
        }
        // ---- pass 2: exponentials against the reference, P over the scores just consumed
        const float mneg = ref_negative(m, sl2);
        const uint64_t mnegx2 = pack2(mneg, mneg);
        uint64_t lsum[4] = {0ull, 0ull, 0ull, 0ull};
        uint32_t pk[16];
        exp32<false, kPolyOf8>(va, sl2x2, mnegx2, lsum, pk, mx4);
        if (kWpt == 2 && !pre) {                       // the other window's keys: probability zero
          const bool right = (lane >> 3) & 1;
#pragma unroll
          for (int i = 0; i < 16; ++i) {
            va[8 * (i >> 2) + (i & 3)] = right ? 0u : pk[i];
            va[8 * (i >> 2) + 4 + (i & 3)] = right ? pk[i] : 0u;
          }
          tmem_st32(tS, va);
        } else {
          tmem_st16(tS, pk);
        }
        if (kWpt != 2 && !pre) {
          tmem_ld32(tS + 32, va);
          tmem_wait_ld(va);
          exp32<false, kPolyOf8>(va, sl2x2, mnegx2, lsum, pk, mx4);
          tmem_st16(tS + 16, pk);
        }
        float a0, a1, b0, b1;
        unpack2(add2(lsum[0], lsum[1]), a0, a1);
        unpack2(add2(lsum[2], lsum[3]), b0, b1);
        l += (a0 + a1) + (b0 + b1);
        // publish P
        tmem_wait_st();
        tc_fence_before();
        mbar_arrive(&bar->p_full[t]);
        if (u == 0) release();         // the previous item's store has long read its staging quarter
      }
      if (!ok) break;
      // ---- epilogue: O / l -> bf16 -> this warp's quarter of the tile's Q buffer (its scores are all complete) -> one TMA store
      ok = warp_wait<kSuspendNs>(&bar->o_full[t], n & 1, &bar->abort_flag, p.status);
      if (!ok) break;
      tc_fence_after();
      const float inv = ref_inverse(m, l);
      const int wx0 = it.x0, wy0 = it.y0 + x * p.box_h + sub_y;           // origin of this warp's sub-box
      const bool store = wx0 < it.x_end && wy0 < it.y_end;                // else none of its rows exists
      unsigned char* stg = smem + (size_t)(2 * t + (n & 1)) * kTileBytes + q4 * 4096;
#pragma unroll 1
      for (int c = 0; c < 2; ++c) {
        uint32_t v[32];
        tmem_ld32(tO + 32 * c, v);
        tmem_wait_ld(v);
        if (store) {
#pragma unroll
          for (int i = 0; i < 4; ++i) {     // 16-byte chunk 4 c + i of this row, at its 128-byte-swizzle position
            const uint4 w = make_uint4(pack_bf16(__uint_as_float(v[8 * i]) * inv, __uint_as_float(v[8 * i + 1]) * inv),
                                       pack_bf16(__uint_as_float(v[8 * i + 2]) * inv, __uint_as_float(v[8 * i + 3]) * inv),
                                       pack_bf16(__uint_as_float(v[8 * i + 4]) * inv, __uint_as_float(v[8 * i + 5]) * inv),
                                       pack_bf16(__uint_as_float(v[8 * i + 6]) * inv, __uint_as_float(v[8 * i + 7]) * inv));
            *reinterpret_cast<uint4*>(stg + lane * 128 + (((4 * c + i) ^ (lane & 7)) << 4)) = w;
          }
        }
      }
      tc_fence_before();
      if (store) {
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
        if (lane == 0) {
          tma_store_4d(&mapO, smem_u32(stg), 0, wx0, wy0, it.bh);   // rows past the grid edge are clipped
          asm volatile("cp.async.bulk.commit_group;" ::: "memory");
        }
      }
      held = n & 1;
      ++n;
    }
    if (ok) release();
    // the staging tile must outlive the last store's reads; wait for the writes as well
    if (lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
  }

  // ================= common teardown =================
  // with prefix tokens this launch overlaps the one ahead of it (their queries) and must not end before it
  if (kPrefix) griddep_wait();
  __syncwarp();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
}

}  // namespace

// Windows of exactly one or two tile boxes (box = window width x 128 / width rows), or of 8 x 8 tokens; at most 16 prefix
// tokens (contiguous inputs only: the prefix rows are found behind a.k and a.v).
bool attn_w4_supported(const AttnArgs& a) {
  if (a.dtype != JV_BF16 || a.D != kD) return false;
  if (a.P > kPreRows || (a.P > 0 && a.strided)) return false;
  const int ww = a.ww;
  if (ww < 1 || ww > 32 || (ww & (ww - 1)) != 0) return false;   // a warp's 32 rows are whole box rows
  const int bh = kTile / ww;
  if (a.wh != bh && a.wh != 2 * bh && !(ww == 8 && a.wh == 8)) return false;
  const int64_t nwin = (int64_t)ceil_div(a.Wg, ww) * ceil_div(a.Hg, a.wh);
  if (nwin * a.BH > 0x7fffffffll) return false;
  return encode_fn() != nullptr;
}

// CTAs of a launch.  Fewer items than SMs: one to a CTA.  With prefix tokens and less than a wave of items, both slots of
// half as many CTAs work, if that leaves the prefix queries' launch SMs of its own: the two run side by side (42 heads
// of 28 x 28 tokens: 16.5 us; behind one another, with the items over all SMs, 20.9).
int attn_w4_ctas(const AttnArgs& a) {
  const int box_w = a.ww * a.wh == 64 ? 2 * a.ww : a.ww, box_h = kTile / box_w;
  const int64_t total = (int64_t)ceil_div(a.Wg, box_w) * ceil_div(a.Hg, 2 * box_h) * a.BH;
  const int sms = device_sm_count();
  if (a.P > 0 && total <= kSlots * sms && total + a.BH > sms) return (int)((total + kSlots - 1) / kSlots);
  return (int)(total < sms ? total : sms);
}

template <bool kPrefix, int kWpt>
cudaError_t launch_w4(const CUtensorMap (&maps)[6], const W4Params& p, int grid, cudaStream_t st) {
  static OncePerDevice smem_opt_in;   // > 48 KB of dynamic shared memory: a per-device function attribute
  const cudaError_t e = smem_opt_in.run([] {
    return cudaFuncSetAttribute(attn_w4_kernel<kPrefix, kWpt>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)Layout<kPrefix>::kBytes);
  });
  if (e != cudaSuccess) return e;
  return launch_programmatic(attn_w4_kernel<kPrefix, kWpt>, dim3(grid), kThreads, Layout<kPrefix>::kBytes, st, maps[0], maps[1], maps[2],
                             maps[3], maps[4], maps[5], p);
}

cudaError_t launch_attn_w4(const AttnArgs& a, int* status, cudaStream_t st) {
  EncodeFn enc = encode_fn();
  if (!enc) return cudaErrorNotSupported;
  const int N = a.P + a.Hg * a.Wg;                     // tokens per (batch, head): prefix tokens, then the grid
  // windows per tile (see the head of this file)
  const int wpt = a.ww * a.wh == 64 ? 2 : a.ww * a.wh == kTile ? 1 : 0;
  const int box_w = wpt == 2 ? 2 * a.ww : a.ww, box_h = kTile / box_w;
  CUtensorMap maps[6];
  // the grid tokens start behind the prefix rows
  const size_t grid0 = (size_t)a.P * kD * 2, igrid0 = (size_t)a.P * (size_t)a.in.tok * 2;
  const void* ptrs[4] = {(const char*)a.q + igrid0, (const char*)a.k + igrid0, (const char*)a.v + igrid0, (char*)a.o + grid0};
  const cuuint64_t dims[4] = {(cuuint64_t)kD, (cuuint64_t)a.Wg, (cuuint64_t)a.Hg, (cuuint64_t)a.BH};
  const cuuint64_t strides[3] = {(cuuint64_t)kD * 2, (cuuint64_t)a.Wg * kD * 2, (cuuint64_t)N * kD * 2};
  // the output is stored per warp: a quarter of the tile's box (32 tokens)
  const cuuint32_t qbox[4] = {(cuuint32_t)kD, (cuuint32_t)box_w, (cuuint32_t)(box_h / 4), 1};
  const cuuint32_t estr[4] = {1, 1, 1, 1};
  // the inputs as (d, x, y, head, batch) with the caller's strides; the output as (d, x, y, batch*head)
  const cuuint64_t idims[5] = {(cuuint64_t)kD, (cuuint64_t)a.Wg, (cuuint64_t)a.Hg, (cuuint64_t)a.H, (cuuint64_t)(a.BH / a.H)};
  const cuuint64_t istrides[4] = {(cuuint64_t)a.in.tok * 2, (cuuint64_t)a.Wg * a.in.tok * 2, (cuuint64_t)a.in.head * 2,
                                  (cuuint64_t)a.in.batch * 2};
  const cuuint32_t ibox[2][5] = {{(cuuint32_t)kD, (cuuint32_t)box_w, (cuuint32_t)box_h, 1, 1},          // a query tile
                                 {(cuuint32_t)kD, (cuuint32_t)box_w, (cuuint32_t)(box_h / 2), 1, 1}};   // 64 keys
  const cuuint32_t iestr[5] = {1, 1, 1, 1, 1};
  for (int i = 0; i < 4; ++i) {
    CUresult r = i < 3 ? enc(&maps[i], CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<void*>(ptrs[i]), idims, istrides, ibox[i > 0],
                             iestr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                             CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE)
                       : enc(&maps[i], CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(ptrs[i]), dims, strides, qbox,
                             estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                             CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return cudaErrorInvalidValue;
  }
  // the P prefix rows of K and V as (d, row, head, batch), a box of 16 rows: rows past P arrive as zeros
  maps[4] = maps[1];
  maps[5] = maps[2];
  if (a.P > 0) {
    const cuuint64_t pdims[4] = {(cuuint64_t)kD, (cuuint64_t)a.P, (cuuint64_t)a.H, (cuuint64_t)(a.BH / a.H)};
    const cuuint64_t pstrides[3] = {(cuuint64_t)a.in.tok * 2, (cuuint64_t)a.in.head * 2, (cuuint64_t)a.in.batch * 2};
    const cuuint32_t pbox[4] = {(cuuint32_t)kD, (cuuint32_t)kPreRows, 1, 1};
    const void* pptrs[2] = {a.k, a.v};
    for (int i = 0; i < 2; ++i) {
      CUresult r = enc(&maps[4 + i], CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(pptrs[i]), pdims, pstrides, pbox,
                       estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                       CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
      if (r != CUDA_SUCCESS) return cudaErrorInvalidValue;
    }
  }
  W4Params p;
  p.P = a.P;
  p.status = status;
  p.gridW = a.Wg;
  p.gridH = a.Hg;
  p.win_w = box_w;
  p.win_h = 2 * box_h;
  p.box_w = box_w;
  p.box_h = box_h;
  p.lg_box_w = 0;
  while ((1 << p.lg_box_w) < box_w) ++p.lg_box_w;
  p.nwx = ceil_div(a.Wg, p.win_w);
  p.nwin = p.nwx * ceil_div(a.Hg, p.win_h);
  p.total = p.nwin * a.BH;
  p.div_nwin = make_fastdiv((uint32_t)p.nwin);
  p.div_nwx = make_fastdiv((uint32_t)p.nwx);
  p.H = a.H;
  p.div_H = make_fastdiv((uint32_t)a.H);
  p.scale_log2 = a.scale * 1.4426950408889634f;
  const int grid = attn_w4_ctas(a);
  if (a.P > 0)
    return wpt == 0 ? launch_w4<true, 0>(maps, p, grid, st) : wpt == 1 ? launch_w4<true, 1>(maps, p, grid, st) : launch_w4<true, 2>(maps, p, grid, st);
  return wpt == 0 ? launch_w4<false, 0>(maps, p, grid, st) : wpt == 1 ? launch_w4<false, 1>(maps, p, grid, st) : launch_w4<false, 2>(maps, p, grid, st);
}

}  // namespace jv
