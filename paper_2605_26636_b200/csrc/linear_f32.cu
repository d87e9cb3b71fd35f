// Linear-attention block on fp32 tensors at head_dim 64 (Sec. 3.2.1, Eq. 2 reordered, Eq. 4): fp32 multiply-adds
// throughout, register-tiled, with the 3 x 3 convolution inside the apply pass.
//
//   lin_f32_state_kernel   per (head, token chunk): KV = relu(K)^T V, z, v-sum -> partial (layout of lin_common.cuh)
//   generator              dwc_generator.cu
//   lin_f32_apply_kernel   per 32 (64) tokens: sums the chunk partials of its head in chunk order, then
//                          o = relu(q) KV / (relu(q).z + eps) + 3 x 3 convolution of V
//
// The arithmetic is small (128 multiply-adds per token and channel); at the sizes fp32 tensors are used at, these
// are chains of short kernels, so each is laid out to have everything it can load in flight before it waits for
// the kernel ahead of it (programmatic launches), and chunks are short (64 tokens and up) so that the chip is filled.
// A thread of the state pass owns 8 x 4 outputs (three 128-bit shared-memory loads per 16 packed multiply-adds), one of the
// apply pass 4 x 4 or 8 x 4.
//
// The shape-generic kernels, which served these calls before: 12 heads, 32 x 32 tokens, with the convolution 265 us
// against 22 us here; 6 heads, 16 x 16 tokens, without it 116 us against 9.7.
#include "f32_common.cuh"
#include "lin_common.cuh"

namespace jv {
namespace {

using namespace f32;
using namespace lin;

constexpr int kTok = 64;         // tokens per tile
constexpr int kThreads = 128;
constexpr int kLdA = kD + 4;     // padded rows of the apply pass
constexpr size_t kStateSmem = (size_t)2 * 2 * kTok * kD * sizeof(float);             // two stages of K and V
constexpr size_t apply_smem(int rows) { return (size_t)(8 * rows + kD) * kLdA * sizeof(float) + kD * sizeof(float); }

__global__ void __launch_bounds__(kThreads)
lin_f32_state_kernel(const float* __restrict__ k, const float* __restrict__ v, float* __restrict__ partial, int N,
                     int chunk_tokens, int state_elems) {
  extern __shared__ __align__(16) float smem_f[];
  griddep_wait();
  griddep_launch_dependents();
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;      // rows a = 8 ty + i, columns e = 4 tx + j of KV
  const int t_begin = blockIdx.x * chunk_tokens, t_end = min(N, t_begin + chunk_tokens);
  const int ntiles = (t_end - t_begin + kTok - 1) / kTok;
  const size_t base = (size_t)blockIdx.y * N * kD;

  auto load_tile = [&](int it) {
    float* ks = smem_f + (it & 1) * 2 * kTok * kD;
    float* vs = ks + kTok * kD;
    if (it < ntiles) {
#pragma unroll
      for (int i = 0; i < kTok / 8; ++i) {
        const int r = 8 * i + ty, t = t_begin + it * kTok + r;
        const bool in = t < t_end;
        const size_t off = base + (size_t)(in ? t : 0) * kD + 4 * tx;
        copy16(ks + r * kD + 4 * tx, k + off, in);
        copy16(vs + r * kD + 4 * tx, v + off, in);
      }
    }
    copy_commit();
  };

  f32x2 acc[8][2];
#pragma unroll
  for (int i = 0; i < 8; ++i) acc[i][0] = acc[i][1] = 0ull;
  float colsum = 0.f;                                             // threads 0..63: z, threads 64..127: v-sum
  load_tile(0);
  load_tile(1);
  for (int it = 0; it < ntiles; ++it) {
    copy_wait<1>();
    __syncthreads();
    const float* ks = smem_f + (it & 1) * 2 * kTok * kD;
    const float* vs = ks + kTok * kD;
#pragma unroll 4
    for (int t = 0; t < kTok; ++t) {
      const float4 ka = *reinterpret_cast<const float4*>(ks + t * kD + 8 * ty);
      const float4 kb = *reinterpret_cast<const float4*>(ks + t * kD + 8 * ty + 4);
      const ulonglong2 vv = *reinterpret_cast<const ulonglong2*>(vs + t * kD + 4 * tx);
      const float kr[8] = {ka.x, ka.y, ka.z, ka.w, kb.x, kb.y, kb.z, kb.w};
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const float x = fmaxf(kr[i], 0.f);
        const f32x2 x2 = pack2(x, x);
        fma2(acc[i][0], x2, vv.x);
        fma2(acc[i][1], x2, vv.y);
      }
    }
    const bool is_k = tid < kD;
    const float* col = is_k ? ks + tid : vs + (tid - kD);
    float s4[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int t = 0; t < kTok; ++t) {
      const float x = col[t * kD];
      s4[t & 3] += is_k ? fmaxf(x, 0.f) : x;
    }
    colsum += (s4[0] + s4[1]) + (s4[2] + s4[3]);
    __syncthreads();                                              // the stage may be refilled
    load_tile(it + 2);
  }
  float* out = partial + ((size_t)blockIdx.y * gridDim.x + blockIdx.x) * state_elems;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const float2 lo = unpack2(acc[i][0]), hi = unpack2(acc[i][1]);
    float* row = out + (8 * ty + i) * kD + 4 * tx;
    *reinterpret_cast<float4*>(row) = make_float4(lo.x, lo.y, hi.x, hi.y);
  }
  out[kOffZ + tid] = colsum;                                      // z (64), then the v-sum (64)
}

// w: kernels [C][3][3] of sample b at w + b * w_batch, or nullptr (no convolution)
// kRows: tokens per thread, 8 kRows per CTA
template <int kRows>
__global__ void __launch_bounds__(kThreads)
lin_f32_apply_kernel(const float* __restrict__ q, const float* __restrict__ v, float* __restrict__ o,
                     const float* __restrict__ partial, const float* __restrict__ w, int w_batch, int H, int P, int Hg, int Wg, int nchunk,
                     int state_elems, float eps) {
  extern __shared__ __align__(16) float smem_f[];
  constexpr int kOwn = 8 * kRows;
  float* qs = smem_f;                                             // relu(q) [kOwn][kLdA]
  float* kv = qs + kOwn * kLdA;                                   // KV [a][e], rows of kLdA
  float* zs = kv + kD * kLdA;
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;      // tokens kRows ty + i, channels 4 tx + j
  const int N = P + Hg * Wg, bh = blockIdx.y, t0 = blockIdx.x * kOwn;
  griddep_launch_dependents();
  const size_t base = (size_t)bh * N * kD;
#pragma unroll
  for (int i = 0; i < kRows; ++i) {                               // q is an input of the call: loaded ahead of the wait
    const int r = 8 * i + ty;
    float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
    if (t0 + r < N) x = __ldg(reinterpret_cast<const float4*>(q + base + (size_t)(t0 + r) * kD + 4 * tx));
    *reinterpret_cast<float4*>(qs + r * kLdA + 4 * tx) = make_float4(fmaxf(x.x, 0.f), fmaxf(x.y, 0.f), fmaxf(x.z, 0.f), fmaxf(x.w, 0.f));
  }
  griddep_wait();                                                 // state pass and generator are complete
  {
    float4 s[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) s[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    float z = 0.f;
    const float* pp = partial + (size_t)bh * nchunk * state_elems;
#pragma unroll 2
    for (int c = 0; c < nchunk; ++c, pp += state_elems) {         // in chunk order: no atomics, bit-reproducible
      if (tid < kD) z += __ldcg(pp + kOffZ + tid);
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const float4 x = __ldcg(reinterpret_cast<const float4*>(pp + (8 * i + ty) * kD + 4 * tx));
        s[i].x += x.x; s[i].y += x.y; s[i].z += x.z; s[i].w += x.w;
      }
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) *reinterpret_cast<float4*>(kv + (8 * i + ty) * kLdA + 4 * tx) = s[i];
    if (tid < kD) zs[tid] = z;
  }
  __syncthreads();
  f32x2 acc[kRows][2];
  float den[kRows];
#pragma unroll
  for (int i = 0; i < kRows; ++i) acc[i][0] = acc[i][1] = 0ull;
  const float4 z4 = *reinterpret_cast<const float4*>(zs + 4 * tx);
#pragma unroll
  for (int i = 0; i < kRows; ++i) {                               // relu(q).z: four terms per lane, summed over 16 lanes
    const float4 x = *reinterpret_cast<const float4*>(qs + (kRows * ty + i) * kLdA + 4 * tx);
    den[i] = fmaf(x.x, z4.x, fmaf(x.y, z4.y, fmaf(x.z, z4.z, x.w * z4.w)));
#pragma unroll
    for (int m = 1; m < 16; m <<= 1) den[i] += __shfl_xor_sync(0xffffffffu, den[i], m);
  }
#pragma unroll 2
  for (int a = 0; a < kD; a += 4) {
    ulonglong2 kk[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) kk[j] = *reinterpret_cast<const ulonglong2*>(kv + (a + j) * kLdA + 4 * tx);
#pragma unroll
    for (int i = 0; i < kRows; ++i) {
      const float4 x = *reinterpret_cast<const float4*>(qs + (kRows * ty + i) * kLdA + a);
      const f32x2 x0 = pack2(x.x, x.x), x1 = pack2(x.y, x.y), x2 = pack2(x.z, x.z), x3 = pack2(x.w, x.w);
      fma2(acc[i][0], x0, kk[0].x);
      fma2(acc[i][1], x0, kk[0].y);
      fma2(acc[i][0], x1, kk[1].x);
      fma2(acc[i][1], x1, kk[1].y);
      fma2(acc[i][0], x2, kk[2].x);
      fma2(acc[i][1], x2, kk[2].y);
      fma2(acc[i][0], x3, kk[3].x);
      fma2(acc[i][1], x3, kk[3].y);
    }
  }
  float r[kRows][4];
#pragma unroll
  for (int i = 0; i < kRows; ++i) {
    const float2 lo = unpack2(acc[i][0]), hi = unpack2(acc[i][1]);
    const float d = den[i] + eps;
    r[i][0] = lo.x / d; r[i][1] = lo.y / d; r[i][2] = hi.x / d; r[i][3] = hi.y / d;
  }
  const int tt = t0 + kRows * ty;                                 // this thread's consecutive tokens
  if (w != nullptr) {
    float wf[4][9];                                               // [channel][tap]
    const float4* wp = reinterpret_cast<const float4*>(w + (size_t)(bh / H) * w_batch + ((size_t)(bh % H) * kD + 4 * tx) * 9);
#pragma unroll
    for (int i = 0; i < 9; ++i) {
      const float4 x = __ldcg(wp + i);
      wf[(4 * i) / 9][(4 * i) % 9] = x.x;
      wf[(4 * i + 1) / 9][(4 * i + 1) % 9] = x.y;
      wf[(4 * i + 2) / 9][(4 * i + 2) % 9] = x.z;
      wf[(4 * i + 3) / 9][(4 * i + 3) % 9] = x.w;
    }
    const int ng = Hg * Wg, g0 = tt - P;                          // first grid token (negative: prefix tokens among them)
    const int xg = g0 >= 0 ? g0 % Wg : g0;                        // its column (negative: a prefix token)
    const float* vg = v + base + (size_t)P * kD + 4 * tx;         // grid token 0
#pragma unroll
    for (int dy = -1; dy <= 1; ++dy) {
      float4 u[kRows + 2];                                        // grid tokens g0 - 1 .. g0 + kRows, one grid row up or down
#pragma unroll
      for (int j = 0; j < kRows + 2; ++j) {
        const int g = g0 + dy * Wg + j - 1;
        u[j] = (g >= 0 && g < ng) ? __ldg(reinterpret_cast<const float4*>(vg + (ptrdiff_t)g * kD)) : make_float4(0.f, 0.f, 0.f, 0.f);
      }
      int x = xg;
#pragma unroll
      for (int i = 0; i < kRows; ++i) {
        // A neighbour in a row outside the grid lies outside [0, ng) and is zero already; one in a
        // column outside the grid would be a token of the row above or below: left out.
#pragma unroll
        for (int dx = 0; dx < 3; ++dx) {
          const bool ok = x >= 0 && (dx == 0 ? x > 0 : dx == 2 ? x + 1 < Wg : true);
          if (ok) {
            const float4 f = u[i + dx];
            const int tap = 3 * (dy + 1) + dx;
            r[i][0] = fmaf(wf[0][tap], f.x, r[i][0]);
            r[i][1] = fmaf(wf[1][tap], f.y, r[i][1]);
            r[i][2] = fmaf(wf[2][tap], f.z, r[i][2]);
            r[i][3] = fmaf(wf[3][tap], f.w, r[i][3]);
          }
        }
        if (++x == Wg) x = 0;
      }
    }
  }
#pragma unroll
  for (int i = 0; i < kRows; ++i)
    if (tt + i < N)
      *reinterpret_cast<float4*>(o + base + (size_t)(tt + i) * kD + 4 * tx) = make_float4(r[i][0], r[i][1], r[i][2], r[i][3]);
}

}  // namespace

bool linear_f32_supported(const LinArgs& a) {
  return a.s.dtype == JV_F32 && a.s.D == kD && !in_strided(a.s) && !(a.dwc && (a.dwc->token_wise || a.dwc->k != 3));
}

cudaError_t launch_linear_f32(const LinArgs& a, const LinPlan& p, cudaStream_t st) {
  const jv_shape& s = a.s;
  const int N = shape_tokens(s), BH = s.B * s.H;
  float* partial = (float*)((char*)a.ws + p.off_partial);
  static OncePerDevice opt_in;
  cudaError_t e = opt_in.run([] {
    return cudaFuncSetAttribute(lin_f32_state_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kStateSmem);
  });
  if (e != cudaSuccess) return e;
  const float* w = nullptr;
  int w_batch = 0;
  if (a.dwc && (e = dwc_static_kernels(a, p, &w, &w_batch, st)) != cudaSuccess) return e;
  e = launch_programmatic(lin_f32_state_kernel, dim3(p.nchunk, BH), kThreads, kStateSmem, st, (const float*)a.k, (const float*)a.v,
                          partial, N, p.chunk_tokens, p.state_elems);
  if (e != cudaSuccess) return e;
  const float* state = partial;
  int nchunk = p.nchunk;
  if (a.dwc && (e = launch_dwc_generator_fast(a, p, partial, false, &state, &nchunk, st)) != cudaSuccess) return e;
  // 32 tokens per CTA: a CTA of 64 has twice the chain, and three of those fit an SM where five do.  64 only where those are one
  // wave and the others just more than one (24 heads of 1024 tokens, with the convolution 33.3 / 35.1 us).  64 / 32 otherwise, chunks
  // as they are now: 6 heads of 256 tokens 11.0 / 9.7 us, 12 of 1024 with the convolution 26.4 / 21.8, 24 of 576 26.4 / 22.9.
  const int64_t sms = device_sm_count();
  const int rows = (int64_t)ceil_div(N, 64) * BH <= 3 * sms && (int64_t)ceil_div(N, 32) * BH > 5 * sms ? 8 : 4;
  return launch_programmatic(rows == 4 ? lin_f32_apply_kernel<4> : lin_f32_apply_kernel<8>, dim3(ceil_div(N, 8 * rows), BH), kThreads,
                             apply_smem(rows), st, (const float*)a.q,
                             (const float*)a.v, (float*)a.o, state, w, w_batch, (int)s.H, (int)s.P, (int)s.Hg, (int)s.Wg, nchunk,
                             p.state_elems, a.eps);
}

}  // namespace jv
