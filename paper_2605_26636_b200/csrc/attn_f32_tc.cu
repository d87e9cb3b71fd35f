// Softmax attention on fp32 tensors at head_dim 64 (Eq. 1, full and windowed, with prefix keys) on the 5th-generation tensor
// cores: an fp32 value is the sum of three bf16 values (its 24 bits), and a product of two such sums is kept to
// the six of its nine terms that reach 2^-24 of it.
//
//   x = x0 + x1 + x2,  x y = x2 y0 + x1 y1 + x0 y2 + x1 y0 + x0 y1 + x0 y0      (small terms first)
//
// Sums stay as they were in fp32 multiply-adds or better: the tensor core's accumulator only takes the terms of ONE
// step of 64 keys (scores: of 64 channels), where the small terms meet before the large ones, so that four additions at
// the size of the result are left; the steps' products with V are added up in fp32 registers, rounded to nearest.
// An infinity in K (or what rounds to one: finite values from bf16's largest on) becomes 2^110 of its sign, so that keys switched off by a
// score of -inf cost little: such a key's score is below -2^69 and weighs nothing against scores within 2^30.  What the
// terms cannot hold, the CTA computes again with fp32 multiply-adds (plain_rows):
//   - a row whose weights or results are no finite numbers (a score of +inf or NaN, no key of weight, infinities in V);
//   - beside infinities in K: a zero of q in such a channel (a score of NaN), values of q beyond 2^25 or below 2^-40 (the bounds above), a row
//     whose largest score is beyond 2^30, a key with two infinities or with other values beyond 2^30;
//   - values of q beyond 2^60, or below 2^-100 but not 0; results below 2^-80 beside values of V below 2^-60 but not 0.  The third term of very
//     small values, or its products, may lie below 2^-126, the normal range, and bits get lost from 2^-110 on.  (What k loses there is
//     below 2^-68 of a score: nothing while the softmax scale is at most 2^40: launch_attn_f32.)
// All of this is looked at where it is cheap: K by the sum of its magnitudes and the issuing warp, V by the results.
//
// One CTA serves 128 query rows of one (batch, head) and window, with its key tiles (64 keys) dealt to two slots: a slot
// has its own four softmax warps (a thread per row), three warps that cut K and V into bf16 planes, MMA issuer and rings, so that
// one slot's softmax runs under the other's products.  Windows of at most 64 tokens go two to a CTA: rows 0-63 and slot 0
// are one window, rows 64-127 and slot 1 the next.
//
// Warp roles (16 warps): 0-7 softmax (slot w / 4); 8-11 and 12-15 serve slots 0 and 1: the first issues the MMAs, three bring K and
// V from global memory into planes in shared memory.  Tensor memory (all 512 columns): two planes of Q (the third is in shared
// memory); per slot two buffers of 64 columns of scores, then of two planes of probabilities, 32 columns of the third plane,
// and 64 of the step's product with V.  The scores of step u + 1 are computed while the softmax works on step u.
//
// What bounds it: the tensor pipe, 48 MMAs of M128 N64 K16 per step (1536 clocks), with the exponentials and the cutting of P, K
// and V (about 1370 issue slots a step and sub-core) right behind; a pair of steps, one per slot, takes 4000 clocks.  A call of one round of CTAs takes
// 10 us for 128 keys (launch, first loads, first step, merge) and 2.4 for every further 128.
// Measured (the kernel of fp32 multiply-adds, attn_f32.cu, in brackets): full attention, 12 heads of 32 x 32 tokens 27.9 us (93.9), 24 of 37 x 37 65.9
// (279), 192 of 1024 309 (1177); 16 x 16 windows, 12 heads of 32 x 32 13.8 (27.3), 96 83.5 (166).  Without the looks at what three terms cannot hold, and with the
// scale in the exponent's multiply-add, 26.6, 64.0, 300; 13.4, 80.  Error against fp64, 2-norm: 1.6e-7 to 2.1e-7
// (2.1e-7 to 5.1e-7) over 6 to 192 heads of 64 to 1400 tokens, with q four times as large 2.3e-7 to 3.1e-7 (3.4e-7 to 6.7e-7).  With terms cut off instead of rounded the
// terms left out all had the product's sign: 2.3e-7 to 2.8e-7.  With one score buffer per slot 33.1 us in place of 26.3; with the third plane of P in a plane of its own
// per buffer there is no tensor memory left.
#include "f32_common.cuh"
#include "tc_common.cuh"

namespace jv {
namespace {

using namespace tc;

constexpr uint32_t kSuspendNs = 4000;          // suspend-time hint of this kernel's barrier waits (tc_common.cuh)
constexpr int kD = 64;
constexpr int kTile = 128;                     // query rows
constexpr int kSub = 64;                       // keys per step
constexpr int kSlots = 2;
constexpr int kStages = 2;                     // of a slot's K ring and of its V ring
constexpr int kPlane = kSub * kD * 2;          // a bf16 plane of a key tile: 8 KB, 128-byte swizzle
constexpr int kStageBytes = 3 * kPlane;
constexpr int kSlotBytes = 2 * kStages * kStageBytes;
constexpr int kWarps = 16, kThreads = kWarps * 32;
constexpr int kWarpSlot = 8;                   // first of the warps that are no softmax warps
constexpr int kConvRows = 11;                  // rows of a key tile per thread: six groups of 16 lanes take rows r0 + 6 i
// Registers: a sub-core holds two softmax warps and two others, of 128 registers each at launch, then of 168 and 88.
constexpr int kRegsLaunch = 128, kRegsSoftmax = 168, kRegsOther = 88;
static_assert(kRegsSoftmax + kRegsOther <= 2 * kRegsLaunch, "register pool of the block");
constexpr uint32_t kTmemCols = 512;
// columns: plane i < 2 of Q at 32 i; slot s from 64 + 224 s on: scores of step u at 64 (u & 1), third plane of P, product
constexpr uint32_t kColSlot = 64, kSlotCols = 224, kColP2 = 128, kColO = 160;
constexpr uint32_t kIdescQK = idesc(kTile, kSub, 0), kIdescPV = idesc(kTile, kD, 1);
// Column of plane i < 2 of the probabilities of keys 16 c .. 16 c + 15, from the step's scores: the planes of 32 keys
// lie over those 32 scores, so that the other half's scores are still there
__host__ __device__ constexpr uint32_t col_p(int i, int c) { return 32 * (c >> 1) + 16 * i + 8 * (c & 1); }

struct Params {
  const float *q, *k, *v;
  float* o;
  int* status;
  int Hg, Wg, P;          // token grid behind P prefix tokens
  int wh, ww, nwx, nwin;  // windows (wh <= Hg, ww <= Wg)
  bool pair;              // two windows to a CTA
  bool overlap;           // the launch ahead is that of the prefix queries of this call
  float scale, sl2;       // softmax scale, and times log2(e)
};

// What a CTA has met.  kSpecial: its rows have to be computed with multiply-adds; kUntame: if there are infinities in K, too; kInf: there are;
// kZero: zeros in Q, which matter if they meet one; kLookV: results below 2^-80, which may come of too small values of V; kUnclear: one of these does
enum : uint32_t { kSpecial = 1, kUntame = 2, kInf = 4, kZero = 8, kLookV = 16, kUnclear = 32 };
struct __align__(8) Barriers {
  uint64_t q_full;
  uint64_t k_full[kSlots][kStages], k_empty[kSlots][kStages], v_full[kSlots][kStages], v_empty[kSlots][kStages];
  uint64_t s_full[kSlots][2], p_full[kSlots], o_full[kSlots];
  uint64_t drain;
  uint32_t tmem_base;
  volatile uint32_t abort_flag;
  uint32_t flags;                              // kSpecial ..
  volatile int k_odd[kSlots][kStages];         // 1 + step of a tile of K with values that are no numbers or beyond 2^60
  uint32_t k_inf[2];                           // channels 32 i .. with an infinity in K
};
constexpr int kOffQ2 = kSlots * kSlotBytes;    // third plane of Q [128][64], 128-byte swizzle
constexpr size_t kSmemTiles = kOffQ2 + kTile * kD * 2;
constexpr size_t kSmemBytes = kSmemTiles + sizeof(Barriers) + 1024;        // + alignment slack
static_assert(kSmemBytes <= 232448, "shared memory of one CTA");
// after its last product a slot's ring takes what the other slot merges: [32 channels / 4][row] 16-byte pieces, then (m, l)
constexpr int kPartBytes = kTile * (kD / 2) * 4;
static_assert(kPartBytes + kTile * 8 <= kSlotBytes, "a slot's half of the output");

// One window: origin, valid extent, and its queries and keys by index (keys: prefix tokens, then the window's own)
struct Window {
  int y0, x0, vw, nq, cnt, P, Wg;
  bool dense;             // consecutive keys are consecutive tokens
  __device__ __forceinline__ Window(const Params& p, int w) : P(p.P), Wg(p.Wg) {
    const int wy = w / p.nwx, wx = w - wy * p.nwx;
    y0 = wy * p.wh;
    x0 = wx * p.ww;
    vw = min(p.ww, p.Wg - x0);
    nq = w < p.nwin ? min(p.wh, p.Hg - y0) * vw : 0;
    cnt = w < p.nwin ? p.P + nq : 0;
    dense = vw == p.Wg;
  }
  __device__ __forceinline__ int key_token(int c) const {
    if (c < P) return c;
    if (dense) return c + y0 * Wg;
    const int g = c - P, y = g / vw;
    return P + (y0 + y) * Wg + x0 + (g - y * vw);
  }
  __device__ __forceinline__ int query_token(int c) const { return key_token(P + c); }
};

// Two fp32 values -> the nearest bf16 of each (packed, first value low); what is left over stays in x (exactly)
__device__ __forceinline__ uint32_t cut2(uint64_t& x) {
  float lo, hi;
  unpack2(x, lo, hi);
  const uint32_t t = pack_bf16(lo, hi);
  x = fma2(pack2(__uint_as_float(t << 16), __uint_as_float(t & 0xffff0000u)), pack2(-1.f, -1.f), x);
  return t;
}
__device__ __forceinline__ uint32_t last2(uint64_t x) {
  float lo, hi;
  unpack2(x, lo, hi);
  return pack_bf16(lo, hi);
}
__device__ __forceinline__ bool no_number(float x) { return !(fabsf(x) < INFINITY); }
// Infinite or no number once one of the values noted is, or exceeds 2^60
__device__ __forceinline__ void note(uint64_t& bad, uint64_t x) { bad = fma2(x, pack2(0x1p67f, 0x1p67f), bad); }
__device__ __forceinline__ bool noted(uint64_t bad) {
  float b0, b1;
  unpack2(bad, b0, b1);
  return no_number(b0 + b1);
}
// The smallest and the largest magnitude of values (largest: NaN is passed over)
__device__ __forceinline__ float min_abs(float m, const float4& x) {
  asm("{\n.reg .f32 a, b;\nabs.f32 a, %1;\nabs.f32 b, %2;\nmin.f32 %0, %0, a, b;\nabs.f32 a, %3;\nabs.f32 b, %4;\nmin.f32 %0, %0, a, b;\n}"
      : "+f"(m) : "f"(x.x), "f"(x.y), "f"(x.z), "f"(x.w));
  return m;
}
__device__ __forceinline__ float max_abs(float m, const float4& x) {
  asm("{\n.reg .f32 a, b;\nabs.f32 a, %1;\nabs.f32 b, %2;\nmax.f32 %0, %0, a, b;\nabs.f32 a, %3;\nabs.f32 b, %4;\nmax.f32 %0, %0, a, b;\n}"
      : "+f"(m) : "f"(x.x), "f"(x.y), "f"(x.z), "f"(x.w));
  return m;
}
constexpr float kSmall = 0x1p-100f;

// Four values in three planes of a ring stage
__device__ __forceinline__ void store3(unsigned char* to, uint64_t a, uint64_t b) {
  uint2 y;
  y.x = cut2(a); y.y = cut2(b);
  *reinterpret_cast<uint2*>(to) = y;
  y.x = cut2(a); y.y = cut2(b);
  *reinterpret_cast<uint2*>(to + kPlane) = y;
  y.x = last2(a); y.y = last2(b);
  *reinterpret_cast<uint2*>(to + 2 * kPlane) = y;
}
__device__ __forceinline__ void tmem_st8(uint32_t taddr, const uint32_t (&r)[8]) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};"
               ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]) : "memory");
}

// Infinities in a tile of K that has just been cut, by the warp that issues its MMAs: two rows to a lane.  planes: the first of three.
// (In the warps that cut, even a branch that is never taken cost 5 %, their loads being in flight there.)
__device__ __forceinline__ void cut_infinities(unsigned char* planes, Barriers* bar, int lane) {
#pragma unroll 1
  for (int row = lane; row < kSub; row += 32) {
    int infs = 0, bigs = 0;                                    // values that are infinite or no number; those and others beyond 2^30
#pragma unroll 4
    for (int c = 0; c < kD / 8; ++c) {
      uint32_t* at = reinterpret_cast<uint32_t*>(planes + row * 128 + ((c ^ (row & 7)) << 4));
      const uint4 y = *reinterpret_cast<const uint4*>(at);
      const uint32_t w[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const uint32_t magnitude = w[j] & 0x7fff7fffu, inf = (magnitude + 0x00800080u) & 0x80008000u;
        bigs += __popc((magnitude + 0x317f317fu) & 0x80008000u);
        if (inf == 0) continue;
        infs += __popc(inf);
        uint32_t z = w[j];
#pragma unroll
        for (int h = 0; h < 32; h += 16)
          if (((magnitude >> h) & 0xffffu) == 0x7f80u) {
            z = (z & ~(0x7fffu << h)) | (0x7680u << h);        // 2^110
            at[j + kPlane / 4] &= ~(0xffffu << h);
            at[j + 2 * (kPlane / 4)] &= ~(0xffffu << h);
            const int ch = 8 * c + 2 * j + (h >> 4);
            atomicOr(&bar->k_inf[ch >> 5], 1u << (ch & 31));
          }
        at[j] = z;
      }
    }
    if (infs) atomicOr(&bar->flags, infs > 1 || bigs > infs ? kInf | kSpecial : kInf);
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  __syncwarp();
}
// The rows of a CTA with fp32 multiply-adds: 16 rows to each of the softmax warps, in tiles of 32 keys (of 64 the rings have no room), the next one on
// its way into shared memory under this one.  A pair's windows have their keys each: four warps to either.  12 heads of 1024 tokens: 163 us with the pass on the
// tensor cores (a warp per row, from global memory: 7.9 ms; the grid of attn_f32.cu, which has more and smaller CTAs: 96).
constexpr int kPlainKeys = 32;
constexpr int kPlainTile = kPlainKeys * f32::kLd;               // floats of a tile of K or V
constexpr int kPlainWarp = kPlainKeys * f32::kLdP;
static_assert((kTile * f32::kLd + kSlots * 4 * kPlainTile + kWarpSlot * kPlainWarp) * 4 <= kSmemTiles, "over the rings");
__device__ __forceinline__ void plain_rows(const Params& p, size_t base, int warp, int lane, float* smem) {
  using namespace f32;
  const int set = p.pair ? warp >> 2 : 0, nw = p.pair ? 4 : kWarpSlot, tx = lane & 15, ty = lane >> 4;
  const Window w(p, p.pair ? 2 * blockIdx.y + set : blockIdx.y);
  if (w.cnt == 0) return;                                       // (a pair's second window that does not exist)
  const int row0 = p.pair ? 16 * (warp & 3) : blockIdx.x * kTile + 16 * warp;     // this warp's first row of the window
  float* qs = smem + 16 * warp * kLd;
  float* kv = smem + kTile * kLd + set * 4 * kPlainTile;        // K, V, K, V
  float* ps = smem + kTile * kLd + kSlots * 4 * kPlainTile + warp * kPlainWarp;
  const int ntiles = (w.cnt + kPlainKeys - 1) / kPlainKeys;
  auto load = [&](int t) {
    float* dst = kv + (t & 1) * 2 * kPlainTile;
    for (int r = 2 * (p.pair ? warp & 3 : warp) + ty; r < kPlainKeys; r += 2 * nw) {
      const bool in = t * kPlainKeys + r < w.cnt;
      const size_t at = base + (size_t)(in ? w.key_token(t * kPlainKeys + r) : 0) * kD + 4 * tx;
      copy16(dst + r * kLd + 4 * tx, p.k + at, in);
      copy16(dst + kPlainTile + r * kLd + 4 * tx, p.v + at, in);
    }
    copy_commit();
  };
  auto sync = [&]() {
    if (!p.pair) asm volatile("bar.sync 1, 256;" ::: "memory");
    else if (set == 0) asm volatile("bar.sync 1, 128;" ::: "memory");
    else asm volatile("bar.sync 2, 128;" ::: "memory");
  };
  for (int r = ty; r < 16; r += 2) {
    const bool in = row0 + r < w.nq;
    copy16(qs + r * kLd + 4 * tx, p.q + base + (size_t)(in ? w.query_token(row0 + r) : 0) * kD + 4 * tx, in);
  }
  load(0);                                                      // (one copy group with Q)
  RowTile<kPlainKeys> x;
  for (int t = 0; t < ntiles; ++t) {
    if (t + 1 < ntiles) {
      load(t + 1);
      copy_wait<1>();
    } else {
      copy_wait<0>();
    }
    sync();
    const float* ks = kv + (t & 1) * 2 * kPlainTile;
    x.scores(qs + 8 * ty * kLd, ks, tx);
    x.softmax(w.cnt - t * kPlainKeys, p.scale, ps, tx, ty);
    __syncwarp();
    x.values(ks + kPlainTile, ps, tx, ty);
    sync();
  }
  x.finish();
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int row = row0 + 8 * ty + i;
    if (row >= w.nq) continue;
    const float4 y = x.row(i);
    const float inv = 1.f / x.l[i];
    *reinterpret_cast<float4*>(p.o + base + (size_t)w.query_token(row) * kD + 4 * tx) = make_float4(y.x * inv, y.y * inv, y.z * inv, y.w * inv);
  }
}

// Behind the CTA's last use of its rings, by the softmax warps: its rows once more, where that is needed
__device__ __forceinline__ void multiply_add(const Params& p, Barriers* bar, uint32_t met, size_t base, int warp, int lane, float* smem) {
  const int set = p.pair ? warp >> 2 : 0, nw = p.pair ? 4 : kWarpSlot, first = 2 * (p.pair ? warp & 3 : warp) + (lane >> 4), c4 = lane & 15;
  bool again = (met & kSpecial) || ((met & kInf) && (met & kUntame));
  const bool look_q = (met & kInf) && (met & kZero), look_v = met & kLookV;
  if (!again && (look_q || look_v)) {
    const Window w(p, p.pair ? 2 * blockIdx.y + set : blockIdx.y);
    const uint32_t inf = bar->k_inf[c4 >> 3] >> (4 * (c4 & 7));                       // of this lane's four channels
    const int row0 = p.pair ? 0 : blockIdx.x * kTile, rows = look_q ? min(p.pair ? kTile / 2 : kTile, w.nq - row0) : 0;
#pragma unroll 4
    for (int r = first; r < rows + (look_v ? w.cnt : 0); r += 2 * nw) {
      const bool is_q = r < rows;
      const float* src = is_q ? p.q + base + (size_t)w.query_token(row0 + r) * kD : p.v + base + (size_t)w.key_token(r - rows) * kD;
      const float4 x = __ldcg(reinterpret_cast<const float4*>(src) + c4);
      const float e[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
      for (int j = 0; j < 4; ++j) again = again || (is_q ? e[j] == 0.f && ((inf >> j) & 1) : e[j] != 0.f && fabsf(e[j]) < 0x1p-60f);
    }
    if (again) atomicOr(&bar->flags, kUnclear);
    asm volatile("bar.sync 1, 256;" ::: "memory");
    again = *reinterpret_cast<volatile uint32_t*>(&bar->flags) & kUnclear;
  }
  if (again) plain_rows(p, base, warp, lane, smem);
}

__global__ void __launch_bounds__(kThreads, 1)
attn_f32_tc_kernel(const Params p) {
  extern __shared__ unsigned char smem_raw[];
  // 1024-byte alignment by an offset from the array itself, so that accesses stay shared-space loads and stores
  unsigned char* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  Barriers* bar = reinterpret_cast<Barriers*>(smem + kSmemTiles);
  const uint32_t sRing = smem_u32(smem);        // slot s: K stages, then V stages, three planes each
  const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
  const int N = p.P + p.Hg * p.Wg;
  const size_t base = (size_t)blockIdx.z * N * kD;

  if (threadIdx.x == 0) {
    mbar_init(&bar->q_full, 256);
    for (int s = 0; s < kSlots; ++s) {
      for (int g = 0; g < kStages; ++g) {
        bar->k_odd[s][g] = 0;
        mbar_init(&bar->k_full[s][g], 96);
        mbar_init(&bar->k_empty[s][g], 1);
        mbar_init(&bar->v_full[s][g], 96);
        mbar_init(&bar->v_empty[s][g], 1);
      }
      mbar_init(&bar->s_full[s][0], 1);
      mbar_init(&bar->s_full[s][1], 1);
      mbar_init(&bar->p_full[s], 128);
      mbar_init(&bar->o_full[s], 1);
    }
    mbar_init(&bar->drain, kSlots);
    bar->abort_flag = 0;
    bar->flags = bar->k_inf[0] = bar->k_inf[1] = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
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

  // What is read and written from here on may belong to the launch ahead; overlap: that one, of the prefix queries, has waited
  // for what came before it, and is waited for at the end.
  if (!p.overlap) griddep_wait();
  griddep_launch_dependents();
  if (threadIdx.x == 0 && *reinterpret_cast<volatile int*>(p.status) != 0) bar->abort_flag = 1;   // an earlier kernel gave up
  __syncthreads();

  const bool skip = bar->abort_flag || (!p.pair && (int)(blockIdx.x * kTile) >= Window(p, blockIdx.y).nq);   // (a small edge window)
  if (!skip) {
    if (warp >= kWarpSlot) asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegsOther));
    if (warp >= kWarpSlot && (warp & 3) == 0) {
      // ================= MMA issuer of one slot =================
      // S(u) = Q K(u)^T, then O = P(u - 1) V(u - 1): one thread's MMAs execute in issue order, so S(u) may lie where P(u - 2) was.
      // The softmax threads take O before they publish the next P.
      const int s = (warp - kWarpSlot) >> 2;
      const Window w(p, p.pair ? 2 * blockIdx.y + s : blockIdx.y);
      const int first = p.pair ? 0 : s, stride = p.pair ? 1 : kSlots;
      const int ntiles = (w.cnt + kSub - 1) / kSub, n = ntiles > first ? (ntiles - first + stride - 1) / stride : 0;
      const uint32_t tS = tmem + kColSlot + s * kSlotCols, tO = tS + kColO;
      const uint32_t ringK = sRing + s * kSlotBytes, ringV = ringK + kStages * kStageBytes;
      constexpr int kA[6] = {2, 1, 0, 1, 0, 0}, kB[6] = {0, 1, 2, 0, 1, 0};        // terms, small ones first
      bool ok = warp_wait<kSuspendNs>(&bar->q_full, 0, &bar->abort_flag, p.status);
      for (int u = 0; u <= n && ok && n > 0; ++u) {
        if (u < n) {
          const int g = u % kStages;
          ok = warp_wait<kSuspendNs>(&bar->k_full[s][g], (u / kStages) & 1, &bar->abort_flag, p.status);
          if (!ok) break;
          if (bar->k_odd[s][g] == u + 1) cut_infinities(smem + s * kSlotBytes + g * kStageBytes, bar, lane);
          tc_fence_after();
          if (elect_one()) {
            const uint64_t dq = smem_desc(sRing + kOffQ2);
#pragma unroll
            for (int t = 0; t < 6; ++t) {
              const uint64_t dk = smem_desc(ringK + g * kStageBytes + kB[t] * kPlane);
#pragma unroll
              for (int c = 0; c < kD / 16; ++c) {
                if (kA[t] == 2) mma_ss_1(tS + 64 * (u & 1), desc_advance(dq, c * 32), desc_advance(dk, c * 32), kIdescQK, (t > 0 || c > 0) ? 1u : 0u);
                else mma_ts_1(tS + 64 * (u & 1), tmem + kA[t] * 32 + c * 8, desc_advance(dk, c * 32), kIdescQK, (t > 0 || c > 0) ? 1u : 0u);
              }
            }
          }
          __syncwarp();
          tc_commit(&bar->s_full[s][u & 1]);
          tc_commit(&bar->k_empty[s][g]);
        }
        if (u > 0) {
          const int g = (u - 1) % kStages;
          const uint32_t tP = tS + 64 * ((u - 1) & 1);
          ok = warp_wait<kSuspendNs>(&bar->v_full[s][g], ((u - 1) / kStages) & 1, &bar->abort_flag, p.status);
          if (ok) ok = warp_wait<kSuspendNs>(&bar->p_full[s], (u - 1) & 1, &bar->abort_flag, p.status);
          if (!ok) break;
          tc_fence_after();
          if (elect_one()) {
#pragma unroll
            for (int t = 0; t < 6; ++t) {
              const uint64_t dv = smem_desc(ringV + g * kStageBytes + kB[t] * kPlane);
#pragma unroll
              for (int c = 0; c < kSub / 16; ++c)
                mma_ts_1(tO, kA[t] == 2 ? tS + kColP2 + 8 * c : tP + col_p(kA[t], c), desc_advance(dv, c * 2048), kIdescPV,
                         (t > 0 || c > 0) ? 1u : 0u);
            }
          }
          __syncwarp();
          tc_commit(&bar->o_full[s]);
          tc_commit(&bar->v_empty[s][g]);
        }
      }
      asm volatile("bar.arrive 2, 320;" ::: "memory");          // all that this warp has met is noted
      // Teardown: every MMA issued so far must have retired before tensor memory is released.
      tc_commit(&bar->drain);
      if (lane == 0) {
        const unsigned long long t0 = globaltimer();
        while (!mbar_try(&bar->drain, 0) && globaltimer() - t0 < kWaitLimitNs) {}
      }
      __syncwarp();
    } else if (warp >= kWarpSlot) {
      // ================= K and V of one slot, cut into planes: a thread takes 4 channels of 11 rows of a tile =================
      const int s = (warp - kWarpSlot) >> 2, cw = (warp & 3) - 1;
      const Window w(p, p.pair ? 2 * blockIdx.y + s : blockIdx.y);
      const int first = p.pair ? 0 : s, stride = p.pair ? 1 : kSlots;
      const int ntiles = (w.cnt + kSub - 1) / kSub;
      const int c4 = lane & 15, hi = lane >> 4;               // rows 2 cw + hi + 6 i (from 64 on: none)
      unsigned char* ring = smem + s * kSlotBytes;
      // token of the row that lanes 16 (j & 1) .. + 15 take as their i = j / 2, looked up by lane j
      auto row_token = [&](int t) -> int {
        const int c = t * kSub + 2 * cw + (lane & 1) + 6 * (lane >> 1);
        return t < ntiles && c < w.cnt ? w.key_token(c) : -1;
      };
      float4 x[kConvRows];
      auto load = [&](int i, const float* src, int tok) {
        const int tk = __shfl_sync(0xffffffffu, tok, 2 * i + hi);
        x[i] = tk >= 0 ? __ldcg(reinterpret_cast<const float4*>(src + base + (size_t)tk * kD + 4 * c4)) : make_float4(0.f, 0.f, 0.f, 0.f);
      };
      bool ok = true;
      int u = 0, tok = row_token(first);
#pragma unroll
      for (int i = 0; i < kConvRows; ++i) load(i, p.k, tok);
      for (int t = first; t < ntiles && ok; t += stride, ++u) {
        const int g = u % kStages, next = row_token(t + stride);
#pragma unroll
        for (int kv = 0; kv < 2; ++kv) {
          ok = warp_wait<kSuspendNs>(kv == 0 ? &bar->k_empty[s][g] : &bar->v_empty[s][g], ((u / kStages) & 1) ^ 1, &bar->abort_flag, p.status);
          if (!ok) break;
          uint64_t bad = 0ull;
          unsigned char* dst = ring + (kv * kStages + g) * kStageBytes + (c4 & 1) * 8;
#pragma unroll
          for (int half = 0; half < 2; ++half) {
#pragma unroll
            for (int i = half * 6; i < 6 + half * (kConvRows - 6); ++i) {
              const int row = 2 * cw + hi + 6 * i;
              unsigned char* to = dst + row * 128 + (((c4 >> 1) ^ (row & 7)) << 4);
              uint64_t a = pack2(x[i].x, x[i].y), b = pack2(x[i].z, x[i].w);
              if (row < kSub) {                                 // (a row past the tile is loaded and not stored)
                if (kv == 0) {
                  note(bad, a);
                  note(bad, b);
                }
                store3(to, a, b);
              }
            }
            // the rows just stored are V's, or the next tile's K's: on their way under the other half
#pragma unroll
            for (int i = half * 6; i < 6 + half * (kConvRows - 6); ++i) load(i, kv == 0 ? p.v : p.k, kv == 0 ? tok : next);
          }
          if (kv == 0 && noted(bad)) bar->k_odd[s][g] = u + 1;
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
          mbar_arrive(kv == 0 ? &bar->k_full[s][g] : &bar->v_full[s][g]);
        }
        tok = next;
      }
    } else {
      // ================= softmax: one thread per query row and slot =================
      asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kRegsSoftmax));
      const int s = warp >> 2, q4 = warp & 3, r = 32 * q4 + lane;
      const uint32_t lane_base = (uint32_t)(q4 << 5) << 16;
      const uint32_t tS = tmem + lane_base + kColSlot + s * kSlotCols, tO = tS + kColO;
      const Window w(p, p.pair ? 2 * blockIdx.y + s : blockIdx.y);               // whose keys
      const Window wq(p, p.pair ? 2 * blockIdx.y + (q4 >> 1) : blockIdx.y);      // whose queries
      const int row = p.pair ? (r & 63) : blockIdx.x * kTile + r;
      const int first = p.pair ? 0 : s, stride = p.pair ? 1 : kSlots;
      const int ntiles = (w.cnt + kSub - 1) / kSub, n = ntiles > first ? (ntiles - first + stride - 1) / stride : 0;
      const int row_w = row - lane;                            // the warp's first row
      const bool live = row_w < wq.nq && (!p.pair || (q4 >> 1) == s);   // (warp-uniform) else nothing of it is wanted here
      // Q: this slot's half of the channels of the row, in three planes
      {
        const bool in = row < wq.nq;
        const float4* src = reinterpret_cast<const float4*>(p.q + base + (size_t)wq.query_token(in ? row : 0) * kD + 32 * s);
        float most = 0.f, least = in ? 1.f : 0.f;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          uint32_t y[3][8];
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const float4 x = in ? __ldcg(src + 4 * h + i) : make_float4(0.f, 0.f, 0.f, 0.f);
            uint64_t a = pack2(x.x, x.y), b = pack2(x.z, x.w);
            most = max_abs(most, x);
            least = min_abs(least, x);
            y[0][2 * i] = cut2(a); y[0][2 * i + 1] = cut2(b);
            y[1][2 * i] = cut2(a); y[1][2 * i + 1] = cut2(b);
            y[2][2 * i] = last2(a); y[2][2 * i + 1] = last2(b);
          }
#pragma unroll
          for (int i = 0; i < 2; ++i) tmem_st8(tmem + lane_base + 32 * i + 16 * s + 8 * h, y[i]);
#pragma unroll
          for (int i = 0; i < 2; ++i)                          // 16-byte chunk 4 s + 2 h + i of the row
            *reinterpret_cast<uint4*>(smem + kOffQ2 + r * 128 + (((4 * s + 2 * h + i) ^ (r & 7)) << 4)) =
                make_uint4(y[2][4 * i], y[2][4 * i + 1], y[2][4 * i + 2], y[2][4 * i + 3]);
        }
        if (in && (least < 0x1p-40f || most > 0x1p25f)) {
          uint32_t met = (most > 0x1p60f ? kSpecial : 0u) | (most > 0x1p25f ? kUntame : 0u);
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const float4 x = __ldcg(src + i);
            const float e[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
            for (int j = 0; j < 4; ++j)
              met |= e[j] == 0.f ? kZero : fabsf(e[j]) < kSmall ? kSpecial : fabsf(e[j]) < 0x1p-40f ? kUntame : 0u;
          }
          atomicOr(&bar->flags, met);
        }
        tmem_wait_st();
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        tc_fence_before();
        mbar_arrive(&bar->q_full);
      }
      const uint64_t sl2x2 = pack2(p.sl2, p.sl2);
      uint64_t o[32];
#pragma unroll
      for (int i = 0; i < 32; ++i) o[i] = 0ull;
      float m = -INFINITY, l = 0.f, alpha = 0.f;               // m: the largest score so far
      // o = o alpha + the product of step u with V, alpha as that step found it
      auto take_o = [&](int u) -> bool {
        if (!warp_wait<kSuspendNs>(&bar->o_full[s], u & 1, &bar->abort_flag, p.status)) return false;
        tc_fence_after();
        if (!live) return true;
        const uint64_t a2 = pack2(alpha, alpha);
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          uint32_t v[32];
          tmem_ld32(tO + 32 * c, v);
          tmem_wait_ld(v);
#pragma unroll
          for (int i = 0; i < 16; ++i)
            o[16 * c + i] = fma2(o[16 * c + i], a2, pack2(__uint_as_float(v[2 * i]), __uint_as_float(v[2 * i + 1])));
        }
        return true;
      };
      bool ok = true;
      for (int u = 0; u < n; ++u) {
        ok = warp_wait<kSuspendNs>(&bar->s_full[s][u & 1], (u >> 1) & 1, &bar->abort_flag, p.status);
        if (!ok) break;
        tc_fence_after();
        const uint32_t tSu = tS + 64 * (u & 1);
        if (!live) {                                   // (waits for the product, too: one arrival in a phase of p_full)
          if (u > 0 && !(ok = take_o(u - 1))) break;
        } else {
          uint32_t v[32];
          const int valid = w.cnt - (first + u * stride) * kSub;      // keys that exist in this tile
          if (valid < kSub) {                          // the scores of the others become -inf in tensor memory
#pragma unroll 1
            for (int c = 0; c < 2; ++c) {
              tmem_ld32(tSu + 32 * c, v);
              tmem_wait_ld(v);
#pragma unroll
              for (int i = 0; i < 32; ++i)
                if (32 * c + i >= valid) v[i] = kNegInf;
              tmem_st32(tSu + 32 * c, v);
            }
            tmem_wait_st();
          }
          float mx4[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
          tmem_ld32(tSu + 32, v);
          tmem_wait_ld(v);
          max32(v, mx4);
          tmem_ld32(tSu, v);
          tmem_wait_ld(v);
          max32(v, mx4);
          const float mn = fmaxf(m, max_of(mx4));
          const float ref = mn == -INFINITY ? 0.f : mn;                // all scores so far are -inf: weight 0, not NaN
          const float alpha_u = ex2((m - ref) * p.sl2);                // exp(-inf) = 0 on the first step
          m = mn;
          const uint64_t nref2 = pack2(-ref, -ref);
          uint64_t sum[2] = {0ull, 0ull};
          // probabilities of 32 keys: two planes over their scores, the third in y2.  The largest score is subtracted before the scale comes in:
          // the exponent of the largest is 0 however large the scores are (rounded products of scores beyond 2^32 are off by 2^7 and more)
          auto half = [&](int h, uint32_t (&y2)[2][8]) {
#pragma unroll
            for (int c = 0; c < 2; ++c) {              // 16 keys at a time
              uint32_t y[2][8];
#pragma unroll
              for (int i = 0; i < 8; ++i) {
                const int e = 16 * c + 2 * i;
                float x0, x1;
                unpack2(mul2(add2(pack2(__uint_as_float(v[e]), __uint_as_float(v[e + 1])), nref2), sl2x2), x0, x1);
                uint64_t pr = pack2(ex2(x0), ex2(x1));
                sum[i & 1] = add2(sum[i & 1], pr);
                y[0][i] = cut2(pr);
                y[1][i] = cut2(pr);
                y2[c][i] = last2(pr);
              }
#pragma unroll
              for (int i = 0; i < 2; ++i) tmem_st8(tSu + col_p(i, 2 * h + c), y[i]);
            }
          };
          uint32_t y2[2][8];
          half(0, y2);
          if (u > 0 && !(ok = take_o(u - 1))) break;   // the last step's product: has had half a step's time
          alpha = alpha_u;
          tmem_st8(tS + kColP2, y2[0]);
          tmem_st8(tS + kColP2 + 8, y2[1]);
          tmem_ld32(tSu + 32, v);
          tmem_wait_ld(v);
          half(1, y2);
          tmem_st8(tS + kColP2 + 16, y2[0]);
          tmem_st8(tS + kColP2 + 24, y2[1]);
          float a0, a1;
          unpack2(add2(sum[0], sum[1]), a0, a1);
          l = fmaf(l, alpha, a0 + a1);
          tmem_wait_st();
        }
        tc_fence_before();
        mbar_arrive(&bar->p_full[s]);
      }
      if (ok && n > 0) ok = take_o(n - 1);
      // The slots' partial results: a slot finishes half of the channels and gives the other half away, through
      // its own ring (which nothing reads any more: its last product has retired, or it never had a tile).
      unsigned char* mine = smem + (size_t)s * kSlotBytes;
      const unsigned char* other = smem + (size_t)(s ^ 1) * kSlotBytes;
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const uint64_t a = s == 0 ? o[16 + 2 * i] : o[2 * i], b = s == 0 ? o[17 + 2 * i] : o[2 * i + 1];
        *reinterpret_cast<ulonglong2*>(mine + (size_t)(i * kTile + r) * 16) = make_ulonglong2(a, b);
      }
      *reinterpret_cast<float2*>(mine + kPartBytes + r * 8) = make_float2(m, l);
      asm volatile("bar.sync 1, 256;" ::: "memory");
      if (ok && row < wq.nq && !bar->abort_flag) {
        const float2 ml = *reinterpret_cast<const float2*>(other + kPartBytes + r * 8);
        const float M = fmaxf(m, ml.x);
        const float f = ex2((m - M) * p.sl2), fo = ex2((ml.x - M) * p.sl2);      // a slot without a key: exp(-inf) = 0
        const float L = fmaf(ml.y, fo, l * f), inv = 1.f / L;
        uint64_t zeros = 0ull;                                                     // or no number, once one of the results is no finite one
        float least = 1.f;
        float4* dst = reinterpret_cast<float4*>(p.o + base + (size_t)wq.query_token(row) * kD + 32 * s);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const float4 y = *reinterpret_cast<const float4*>(other + (size_t)(i * kTile + r) * 16);
          float x0, x1, x2, x3;
          unpack2(s == 0 ? o[2 * i] : o[16 + 2 * i], x0, x1);
          unpack2(s == 0 ? o[2 * i + 1] : o[17 + 2 * i], x2, x3);
          const float4 z = make_float4(fmaf(y.x, fo, x0 * f) * inv, fmaf(y.y, fo, x1 * f) * inv, fmaf(y.z, fo, x2 * f) * inv,
                                       fmaf(y.w, fo, x3 * f) * inv);
          dst[i] = z;
          zeros = fma2(pack2(z.x, z.y), 0ull, fma2(pack2(z.z, z.w), 0ull, zeros));
          least = min_abs(least, z);
        }
        float z0, z1;
        unpack2(zeros, z0, z1);
        const uint32_t met = (!(L < INFINITY) || no_number(z0 + z1) ? kSpecial : 0u) | (least < 0x1p-80f ? kLookV : 0u) | (!(fabsf(M) < 0x1p30f) ? kUntame : 0u);
        if (met) atomicOr(&bar->flags, met);
      }
      // (In here the compiler has the softmax warps' registers; behind the roles' end it made the whole kernel 5 % slower.)
      asm volatile("bar.sync 2, 320;" ::: "memory");
      const uint32_t met = *reinterpret_cast<volatile uint32_t*>(&bar->flags);
      if (met && !bar->abort_flag) multiply_add(p, bar, met, base, warp, lane, reinterpret_cast<float*>(smem));
    }
  }
  __syncwarp();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
  if (p.overlap) griddep_wait();
}

}  // namespace

cudaError_t launch_attn_f32_tc(const AttnArgs& a, bool overlap, int* status, cudaStream_t st) {
  static OncePerDevice opt_in;
  const cudaError_t e = opt_in.run(
      [] { return cudaFuncSetAttribute(attn_f32_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemBytes); });
  if (e != cudaSuccess) return e;
  Params p;
  p.q = (const float*)a.q;
  p.k = (const float*)a.k;
  p.v = (const float*)a.v;
  p.o = (float*)a.o;
  p.status = status;
  p.Hg = a.Hg;
  p.Wg = a.Wg;
  p.P = a.P;
  p.wh = a.wh < a.Hg ? a.wh : a.Hg;
  p.ww = a.ww < a.Wg ? a.ww : a.Wg;
  p.nwx = ceil_div(a.Wg, p.ww);
  p.nwin = p.nwx * ceil_div(a.Hg, p.wh);
  p.pair = p.wh * p.ww <= kTile / 2 && p.nwin > 1;
  p.overlap = overlap;
  p.scale = a.scale;
  p.sl2 = a.scale * 1.4426950408889634f;
  const dim3 grid = p.pair ? dim3(1, ceil_div(p.nwin, 2), a.BH) : dim3(ceil_div(p.wh * p.ww, kTile), p.nwin, a.BH);
  return launch_programmatic(attn_f32_tc_kernel, grid, kThreads, kSmemBytes, st, p);
}

}  // namespace jv
