// Packed fp32 arithmetic and asynchronous copies of the fp32 kernels; the row tiles of fp32 attention on multiply-adds.
// sm_100 issues two fp32 multiply-adds of a register pair as one instruction (fma.rn.f32x2).  Internal.
#pragma once

#include "common.cuh"

namespace jv {
namespace f32 {

using f32x2 = unsigned long long;   // two fp32 in one 64-bit register pair

__device__ __forceinline__ void fma2(f32x2& d, f32x2 a, f32x2 b) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b));
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
  f32x2 d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ f32x2 pack2(float lo, float hi) {
  f32x2 d;
  asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(lo), "f"(hi));
  return d;
}
__device__ __forceinline__ float2 unpack2(f32x2 a) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(a));
  return r;
}
// 16 bytes global -> shared; in = false writes zeros and reads nothing
__device__ __forceinline__ void copy16(float* dst, const float* src, bool in) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src),
               "r"(in ? 16 : 0) : "memory");
}
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int kPending>
__device__ __forceinline__ void copy_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(kPending) : "memory"); }


// ---- attention: 16 query rows of a warp against tiles of kKeys keys, head_dim 64 ----------------
// Lane (tx, ty) = (lane % 16, lane / 16) owns rows 8 ty .. 8 ty + 7: of the scores the keys tx + 16 j, of the output the channels
// 4 tx .. 4 tx + 3.  Rows of Q, K and V lie kLd floats apart in shared memory, the probabilities by key, kLdP floats apart.
constexpr int kDim = 64;
constexpr int kRowsWarp = 16;    // query rows per warp
constexpr int kLd = 68;          // floats per shared-memory row: 16-byte reads of 8 consecutive rows touch all banks
constexpr int kLdP = 20;         // floats per key of the transposed probabilities (16 rows): 16-byte writes of 8 keys likewise

template <int kKeys>
struct RowTile {
  static constexpr int kJ = kKeys / 16;
  float m[8], l[8];              // maximum and, of this lane's keys, sum
  f32x2 acc[4][4];               // rows 2 i and 2 i + 1, channel 4 tx + e
  f32x2 s2[8][kJ];               // scores: even and odd channels

  __device__ __forceinline__ RowTile() {
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      m[i] = -INFINITY;
      l[i] = 0.f;
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int e = 0; e < 4; ++e) acc[i][e] = 0ull;
  }
  // qr: row 8 ty of Q
  __device__ __forceinline__ void scores(const float* qr, const float* ks, int tx) {
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
      for (int j = 0; j < kJ; ++j) s2[i][j] = 0ull;
#pragma unroll 4
    for (int c = 0; c < kDim; c += 4) {
      ulonglong2 kk[kJ];
#pragma unroll
      for (int j = 0; j < kJ; ++j) kk[j] = *reinterpret_cast<const ulonglong2*>(ks + (tx + 16 * j) * kLd + c);
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const ulonglong2 qq = *reinterpret_cast<const ulonglong2*>(qr + i * kLd + c);
#pragma unroll
        for (int j = 0; j < kJ; ++j) {
          fma2(s2[i][j], qq.x, kk[j].x);
          fma2(s2[i][j], qq.y, kk[j].y);
        }
      }
    }
  }
  // Probabilities into the warp's buffer ps, the output so far against the new maxima; valid: keys that exist from this tile on
  __device__ __forceinline__ void softmax(int valid, float scale, float* ps, int tx, int ty) {
    const bool ragged = valid < kKeys;
#pragma unroll
    for (int h = 0; h < 2; ++h) {                            // four rows at a time
      float p[kJ][4], alpha[4];                              // [key][row]
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const int i = 4 * h + r;
        float s[kJ];
#pragma unroll
        for (int j = 0; j < kJ; ++j) {
          const float2 e = unpack2(s2[i][j]);
          s[j] = (e.x + e.y) * scale;
          if (ragged && tx + 16 * j >= valid) s[j] = -INFINITY;
        }
        float mx = fmaxf(s[0], s[1]);
        if (kJ == 4) mx = fmaxf(mx, fmaxf(s[2 % kJ], s[3 % kJ]));
#pragma unroll
        for (int w = 1; w < 16; w <<= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, w));
        const float mn = fmaxf(m[i], mx);
        const float ref = mn == -INFINITY ? 0.f : mn;        // all scores so far are -inf: weight 0, not NaN
        alpha[r] = expf(m[i] - ref);                         // exp(-inf) = 0 on the first tile
        m[i] = mn;
        float sum = 0.f;
#pragma unroll
        for (int j = 0; j < kJ; ++j) {
          p[j][r] = expf(s[j] - ref);
          sum += p[j][r];
        }
        l[i] = fmaf(l[i], alpha[r], sum);
      }
#pragma unroll
      for (int j = 0; j < kJ; ++j)
        *reinterpret_cast<float4*>(ps + (tx + 16 * j) * kLdP + ty * 8 + 4 * h) = make_float4(p[j][0], p[j][1], p[j][2], p[j][3]);
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        const f32x2 a2 = pack2(alpha[2 * r], alpha[2 * r + 1]);
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[2 * h + r][e] = mul2(acc[2 * h + r][e], a2);
      }
    }
  }
  __device__ __forceinline__ void values(const float* vs, const float* ps, int tx, int ty) {
#pragma unroll 8
    for (int c = 0; c < kKeys; ++c) {
      const float4 v4 = *reinterpret_cast<const float4*>(vs + c * kLd + 4 * tx);
      const ulonglong2 pa = *reinterpret_cast<const ulonglong2*>(ps + c * kLdP + ty * 8);
      const ulonglong2 pb = *reinterpret_cast<const ulonglong2*>(ps + c * kLdP + ty * 8 + 4);
      const f32x2 vv[4] = {pack2(v4.x, v4.x), pack2(v4.y, v4.y), pack2(v4.z, v4.z), pack2(v4.w, v4.w)};
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        fma2(acc[0][e], pa.x, vv[e]);
        fma2(acc[1][e], pa.y, vv[e]);
        fma2(acc[2][e], pb.x, vv[e]);
        fma2(acc[3][e], pb.y, vv[e]);
      }
    }
  }
  // behind the last tile: l is the whole row's
  __device__ __forceinline__ void finish() {
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
      for (int w = 1; w < 16; w <<= 1) l[i] += __shfl_xor_sync(0xffffffffu, l[i], w);
  }
  __device__ __forceinline__ float4 row(int i) const {       // this lane's four channels of row i, not divided by l
    float x[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const float2 y = unpack2(acc[i / 2][e]);
      x[e] = i % 2 ? y.y : y.x;
    }
    return make_float4(x[0], x[1], x[2], x[3]);
  }
};

}  // namespace f32
}  // namespace jv
