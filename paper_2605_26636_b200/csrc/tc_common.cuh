// Device and host helpers shared by the tcgen05 kernels (attention, projections): mbarrier waits
// with a time limit, TMA copies, tcgen05 issue / tensor-memory access wrappers, shared-memory and
// instruction descriptors, the softmax building blocks, and the tensor-map encoder entry point.
// Internal; every function is inline.
#pragma once

#include <cuda.h>

#include "common.cuh"

namespace jv {
namespace tc {

constexpr unsigned long long kWaitLimitNs = 2000000000ull;   // 2 s: limit of every barrier wait

// Division by a run-time constant without a divide: q = (umulhi(n, mul) + n) >> shr, exact for
// 0 <= n < 2^31 (mul = floor(2^32 (2^shr - d) / d) + 1, shr = ceil(log2 d)).
struct FastDiv {
  uint32_t mul, shr, d;
};
inline FastDiv make_fastdiv(uint32_t d) {
  uint32_t l = 0;
  while ((1ull << l) < d) ++l;
  return FastDiv{(uint32_t)(((1ull << 32) * ((1ull << l) - d)) / d + 1), l, d};
}
__device__ __forceinline__ int fdiv(int n, const FastDiv& f) { return (int)((__umulhi((uint32_t)n, f.mul) + (uint32_t)n) >> f.shr); }

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ unsigned long long globaltimer() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ bool mbar_try(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n.reg .pred p;\n"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      "selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok) : "r"(smem_u32(bar)), "r"(parity) : "memory");
  return ok != 0;
}
// Non-blocking test of a phase: used to take a barrier's round trip off the critical path
// (test early, consume the answer later, fall back to mbar_wait if it was not yet complete).
__device__ __forceinline__ bool mbar_test(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n.reg .pred p;\n"
      "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      "selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok) : "r"(smem_u32(bar)), "r"(parity) : "memory");
  return ok != 0;
}
// The same test with a suspend-time hint: the thread may sleep in the barrier unit for up to that many
// nanoseconds and is woken when the phase completes, instead of coming back after the (short) default
// limit to spin through the loop around it.  A waiting warp then costs the sub-core it shares with
// working warps fewer issue slots: worth 2.4 % on full attention, whose softmax warps are bound by
// issue slots; the linear block's short kernels lost 1 % to it and wait without the hint.
template <uint32_t kHintNs>
__device__ __forceinline__ bool mbar_try_hint(uint64_t* bar, uint32_t parity) {
  if (kHintNs == 0) return mbar_try(bar, parity);
  uint32_t ok;
  asm volatile(
      "{\n.reg .pred p;\n"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n"
      "selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok) : "r"(smem_u32(bar)), "r"(parity), "r"(kHintNs) : "memory");
  return ok != 0;
}
// Bounded wait.  Returns false (after flagging the status word and the CTA abort flag)
// if the phase did not complete within limit_ns or another role already aborted.
// kHintNs > 0: every try may suspend the thread for up to that long (see mbar_try_hint).
template <uint32_t kHintNs = 0>
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, volatile uint32_t* abort_flag, int* status,
                                          unsigned long long limit_ns = kWaitLimitNs) {
  if (mbar_try(bar, parity)) return true;
  constexpr uint32_t kCheckMask = kHintNs >= 1000 ? 15u : 63u;   // tries between looks at the clock and the abort flag
  unsigned long long t0 = 0;
  for (uint32_t spin = 0;; ++spin) {
    if (mbar_try_hint<kHintNs>(bar, parity)) return true;
    if ((spin & kCheckMask) == kCheckMask) {
      if (*abort_flag) return false;
      const unsigned long long now = globaltimer();
      if (t0 == 0) t0 = now;
      else if (now - t0 > limit_ns) {
        *abort_flag = 1;
        atomicOr(status, kStatusTimeout);
        return false;
      }
    }
  }
}

// The same for a whole converged warp, with a warp-uniform outcome.
template <uint32_t kHintNs = 0>
__device__ __forceinline__ bool warp_wait(uint64_t* bar, uint32_t parity, volatile uint32_t* abort_flag, int* status) {
  return __all_sync(0xffffffffu, mbar_wait<kHintNs>(bar, parity, abort_flag, status));
}
__device__ __forceinline__ bool warp_wait_limit(uint64_t* bar, uint32_t parity, volatile uint32_t* abort_flag, int* status,
                                                unsigned long long limit_ns) {
  return __all_sync(0xffffffffu, mbar_wait<0>(bar, parity, abort_flag, status, limit_ns));
}

// Brings a tensor map into the descriptor cache: by one thread, ahead of the wait for the launch before, so that the first copies
// need not fetch theirs (a launch's parameters are new memory every time).  Six layers of 6 heads on 37 x 37 tokens 84.8 -> 84.2 us, three
// of 384 heads on 16 x 16 tokens 69.6 -> 69.4; long launches the same.
__device__ __forceinline__ void prefetch_map(const CUtensorMap* map) {
  asm volatile("prefetch.tensormap [%0];" ::"l"(map) : "memory");
}

__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, uint64_t* bar, int c0, int c1) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
      ::"r"(dst), "l"(map), "r"(smem_u32(bar)), "r"(c0), "r"(c1) : "memory");
}
__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* map, uint64_t* bar, int c0, int c1, int c2) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];"
      ::"r"(dst), "l"(map), "r"(smem_u32(bar)), "r"(c0), "r"(c1), "r"(c2) : "memory");
}
__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap* map, uint64_t* bar, int c0, int c1,
                                            int c2, int c3) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], [%2];"
      ::"r"(dst), "l"(map), "r"(smem_u32(bar)), "r"(c0), "r"(c1), "r"(c2), "r"(c3) : "memory");
}
__device__ __forceinline__ void tma_load_5d(uint32_t dst, const CUtensorMap* map, uint64_t* bar, int c0, int c1,
                                            int c2, int c3, int c4) {
  asm volatile(
      "cp.async.bulk.tensor.5d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6, %7}], [%2];"
      ::"r"(dst), "l"(map), "r"(smem_u32(bar)), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(c4) : "memory");
}
__device__ __forceinline__ void tma_store_3d(const CUtensorMap* map, uint32_t src, int c0, int c1, int c2) {
  asm volatile("cp.async.bulk.tensor.3d.global.shared::cta.tile.bulk_group [%0, {%2, %3, %4}], [%1];"
               ::"l"(map), "r"(src), "r"(c0), "r"(c1), "r"(c2) : "memory");
}

// ---- tcgen05 wrappers -------------------------------------------------------------
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
// One lane of a converged warp (the same one every time for a full warp).
__device__ __forceinline__ bool elect_one() {
  uint32_t pred;
  asm volatile("{\n.reg .pred p;\nelect.sync _|p, 0xffffffff;\nselp.u32 %0, 1, 0, p;\n}\n" : "=r"(pred));
  return pred != 0;
}
// The tcgen05 issue wrappers below are called by a whole converged warp; one elected lane issues.
__device__ __forceinline__ void tc_commit(uint64_t* bar) {
  if (elect_one())
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar)) : "memory");
}
// D[tmem] (+)= A[smem] * B[smem], to be called by ONE lane (the caller holds the election): a run of MMAs issued back to
// back by one thread, without an election and a branch around each of them.
__device__ __forceinline__ void mma_ss_1(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n"
      ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(acc) : "memory");
}
__device__ __forceinline__ void mma_ts_1(uint32_t d_tmem, uint32_t a_tmem, uint64_t bdesc, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}\n"
      ::"r"(d_tmem), "r"(a_tmem), "l"(bdesc), "r"(idesc), "r"(acc) : "memory");
}
// A descriptor moved by `bytes` (a multiple of 16) within its tile: the start-address field counts 16-byte units.
__device__ __forceinline__ uint64_t desc_advance(uint64_t desc, uint32_t bytes) { return desc + (bytes >> 4); }
// D[tmem] (+)= A[tmem] * B[smem]
__device__ __forceinline__ void mma_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t bdesc, uint32_t idesc, uint32_t acc) {
  if (elect_one())
  asm volatile(
      "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}\n"
      ::"r"(d_tmem), "r"(a_tmem), "l"(bdesc), "r"(idesc), "r"(acc) : "memory");
}
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
      "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
        "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
        "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tmem_st32(uint32_t taddr, const uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "
      "{%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,"
      "%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};"
      ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
        "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]),
        "r"(r[16]), "r"(r[17]), "r"(r[18]), "r"(r[19]), "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]),
        "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]), "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31])
      : "memory");
}
// Two stores of eight registers: a store's operands are consecutive registers, and the shorter runs leave the allocator
// fewer moves to make (full attention, 128 heads of 4096 tokens: 548 us, with one store of sixteen 552).
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t (&r)[16]) {
#pragma unroll
  for (int i = 0; i < 16; i += 8)
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};"
                 ::"r"(taddr + i), "r"(r[i]), "r"(r[i + 1]), "r"(r[i + 2]), "r"(r[i + 3]), "r"(r[i + 4]), "r"(r[i + 5]),
                 "r"(r[i + 6]), "r"(r[i + 7]) : "memory");
}
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
// Waits for this thread's outstanding tensor-memory loads.  The registers of the load are
// threaded through the statement so that no use of them can be scheduled ahead of the wait.
__device__ __forceinline__ void tmem_wait_ld(uint32_t (&r)[32]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                 "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15]),
                 "+r"(r[16]), "+r"(r[17]), "+r"(r[18]), "+r"(r[19]), "+r"(r[20]), "+r"(r[21]), "+r"(r[22]), "+r"(r[23]),
                 "+r"(r[24]), "+r"(r[25]), "+r"(r[26]), "+r"(r[27]), "+r"(r[28]), "+r"(r[29]), "+r"(r[30]), "+r"(r[31])
               :: "memory");
}

__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  uint32_t r;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
  return r;
}
// the largest; no number if one of them is none
__device__ __forceinline__ float max3(float a, float b, float c) {
  float d;
  asm("max.NaN.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}
// Two fp32 values in one 64-bit register: the packed fp32x2 arithmetic of sm_100.
__device__ __forceinline__ uint64_t pack2(float lo, float hi) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void unpack2(uint64_t v, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}

// ---- softmax building blocks: 32 scores of one query row at a time -------------------
constexpr uint32_t kNegInf = 0xff800000u;
__device__ __forceinline__ void max32(const uint32_t (&v)[32], float (&mx)[4]) {
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int u = 0; u < 4; ++u)
      mx[u] = max3(mx[u], __uint_as_float(v[8 * i + 2 * u]), __uint_as_float(v[8 * i + 2 * u + 1]));
}
__device__ __forceinline__ float max_of(const float (&mx)[4]) { return max3(max3(mx[0], mx[1], mx[2]), mx[3], mx[3]); }

// The running reference of a row's exponentials.  A score of +inf or no number makes the row no number.  The exponentials do not
// see to that (the polynomial ones below give 2^-126 for it), so the reference does: such a maximum always moves it, and what has been
// summed up is then multiplied by no number.
__device__ __forceinline__ bool ref_moves(float mx, float m, float lazy) { return !(mx <= m + lazy); }
// factor for what has been summed up against reference m when mx (> m, or no number) takes its place; 0 for m = -inf
__device__ __forceinline__ float ref_scale(float m, float mx, float sl2) { return ex2((m - mx) * sl2) + (mx - mx); }
// m = -inf: all scores so far are -inf, and weigh 0 or 2^-126 against any other
__device__ __forceinline__ float ref_negative(float m, float sl2) { return m == -INFINITY ? 0.f : -m * sl2; }
// a row without any key of weight is no number
__device__ __forceinline__ float ref_inverse(float m, float l) { return m == -INFINITY ? __uint_as_float(0x7fc00000u) : 1.f / l; }

// exp2 on the FMA pipe, for part of the scores (the MUFU unit, 16 results per clock and SM,
// is the tightest resource of softmax attention at head_dim 64).  x = n + f with n = round(x),
// f in [-0.5, 0.5]; 2^f by a degree-3 minimax polynomial (relative error 7.5e-5, well below
// the bf16 rounding of P) or of degree 4 (2.6e-6); n goes straight into the exponent field.  Valid for x in [-126, 126]; below and for no number: 2^-126.
constexpr float kPolyC0 = 0.9999280571937561f, kPolyC1 = 0.6932609677314758f;
constexpr float kPolyC2 = 0.2426111251115799f, kPolyC3 = 0.0551716685295105f;
constexpr float kPoly4C0 = 0.9999992614457123f, kPoly4C1 = 0.6931218147366893f, kPoly4C2 = 0.24024744827863667f;
constexpr float kPoly4C3 = 0.055917860319387246f, kPoly4C4 = 0.009570101911169622f;
constexpr float kRoundMagic = 12582912.f;   // 1.5 * 2^23: adding it leaves round(x) in the low mantissa bits
template <int kDeg>
__device__ __forceinline__ void exp2_poly2(uint64_t x, float& p0, float& p1) {
  float x0, x1;
  unpack2(x, x0, x1);
  x = pack2(fmaxf(x0, -126.f), fmaxf(x1, -126.f));
  const uint64_t t = add2(x, pack2(kRoundMagic, kRoundMagic));
  const uint64_t n = add2(t, pack2(-kRoundMagic, -kRoundMagic));
  const uint64_t f = fma2(n, pack2(-1.f, -1.f), x);
  uint64_t q;
  if (kDeg == 3) {
    q = fma2(f, pack2(kPolyC3, kPolyC3), pack2(kPolyC2, kPolyC2));
    q = fma2(q, f, pack2(kPolyC1, kPolyC1));
    q = fma2(q, f, pack2(kPolyC0, kPolyC0));
  } else {
    q = fma2(f, pack2(kPoly4C4, kPoly4C4), pack2(kPoly4C3, kPoly4C3));
    q = fma2(q, f, pack2(kPoly4C2, kPoly4C2));
    q = fma2(q, f, pack2(kPoly4C1, kPoly4C1));
    q = fma2(q, f, pack2(kPoly4C0, kPoly4C0));
  }
  float q0, q1, t0, t1;
  unpack2(q, q0, q1);
  unpack2(t, t0, t1);
  p0 = __uint_as_float(__float_as_uint(q0) + (__float_as_uint(t0) << 23));
  p1 = __uint_as_float(__float_as_uint(q1) + (__float_as_uint(t1) << 23));
}

// p = exp2(s * sl2 + mneg) for 32 scores; adds them into four packed partial sums and packs
// them to bf16 pairs (even key in the low half).  kTrack also folds the scores into mx; of every 8
// score pairs, kPolyOf8 take the polynomial path, of degree kDeg.
template <bool kTrack, int kPolyOf8, int kDeg = 3>
__device__ __forceinline__ void exp32(const uint32_t (&v)[32], uint64_t sl2x2, uint64_t mnegx2, uint64_t (&lsum)[4],
                                      uint32_t (&pk)[16], float (&mx)[4]) {
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    const float s0 = __uint_as_float(v[2 * i]), s1 = __uint_as_float(v[2 * i + 1]);
    if (kTrack) mx[i & 3] = max3(mx[i & 3], s0, s1);
    const uint64_t x = fma2(pack2(s0, s1), sl2x2, mnegx2);
    float p0, p1;
    if ((i & 7) < kPolyOf8) {
      exp2_poly2<kDeg>(x, p0, p1);
    } else {
      float x0, x1;
      unpack2(x, x0, x1);
      p0 = ex2(x0);
      p1 = ex2(x1);
    }
    lsum[i & 3] = add2(lsum[i & 3], pack2(p0, p1));
    pk[i] = pack_bf16(p0, p1);
  }
}

// Shared-memory matrix descriptors (128-byte swizzle; 8-row groups 1024 bytes apart).
//   K-major operand  ([rows][64 bf16], used for Q and K): advance 32 bytes per K step of 16.
//   MN-major operand ([keys][64 bf16] used as B = V):      advance 2048 bytes per K step of 16 keys.
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr) {
  return (uint64_t)((addr & 0x3FFFFu) >> 4) | (1ull << 16) /* LBO (unused) */ | (64ull << 32) /* SBO = 1024 B */ |
         (1ull << 46) /* descriptor version */ | (2ull << 61) /* SWIZZLE_128B */;
}
// Instruction descriptor, kind::f16: D fp32, A and B bf16.
constexpr uint32_t idesc(uint32_t M, uint32_t N, uint32_t b_mn_major, uint32_t a_mn_major = 0) {
  return (1u << 4) | (1u << 7) | (1u << 10) | (a_mn_major << 15) | (b_mn_major << 16) | ((N >> 3) << 17) | ((M >> 4) << 24);
}
// ---- host side: cuTensorMapEncodeTiled through the runtime's driver entry point lookup ----
typedef CUresult (*EncodeFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                             const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                             CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

inline EncodeFn encode_fn() {
  static EncodeFn fn = nullptr;
  if (!fn) {
    void* ptr = nullptr;
    cudaDriverEntryPointQueryResult qres;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &ptr, cudaEnableDefault, &qres) != cudaSuccess ||
        qres != cudaDriverEntryPointSuccess)
      return nullptr;
    fn = (EncodeFn)ptr;
  }
  return fn;
}

}  // namespace tc
}  // namespace jv
