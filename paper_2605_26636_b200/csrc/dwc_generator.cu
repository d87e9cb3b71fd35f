// Kernel generator of the squeeze dynamic convolution (Sec. 3.2.1), head_dim 64:
//
//   mean[b][c]   = (v-sums of the state pass, summed in chunk order) / N
//   hidden[b][r] = SiLU(b1[r] + sum_c W1[r][c] mean[b][c])             gen_hidden_kernel
//   w[b][t]      = b2[t] + sum_r W2[t][r] hidden[b][r]                 gen_out_kernel
//
// It sits on the critical path between the state pass and the apply pass, so what bounds it is latency: round trips
// to L2, and the weights, which a large call has flushed to HBM.  Both kernels have their first weights on the way (inputs
// of the call) before they wait for the grid ahead of them, and everything else they load in flight together.
// (One kernel for both layers, hidden formed by a cluster of eight CTAs, saved the launch but lost more in the
// exchange of the partial sums through distributed shared memory: 10.8 us against 9.7 for 8 samples of 1024 channels.)
//
// Where a head has three chunks or more, blocks beside the hidden layer's sum them (in chunk order) into the head's state, off
// the critical path, for whoever reads the state behind the generator: the apply pass read the chunks one round trip
// after another at its start (1 x 16 heads of 128 x 128 tokens, 16 chunks: 62.0 us for the block, 50.0 so; 2 x 12 heads of 64 x 128,
// 11 chunks: 50.0 and 41.8).
//
// The rows of up to kGenPrefix prefix tokens, which the convolution does not see, are work of the same kind (a few
// products with a head's summed state): blocks behind the output layer's own take them.
#include "lin_common.cuh"

namespace jv {
namespace {

using namespace lin;

constexpr int kThreads = 256;                         // of the hidden layer
constexpr int kThreadsOut = 128;                      // of the output layer
constexpr int kRowsPass = kThreadsOut / 8;            // eight lanes per row of W2
constexpr int kRows = 2;                              // up to this many rows of W2 per thread
constexpr int kAGroups = kThreadsOut / kD;            // prefix rows: groups of threads over the rows of KV
constexpr int kTileC = 1024;                          // channels per pass over the hidden layer
constexpr size_t kMaxSmem = 48 * 1024;                // (no opt-in needed; small enough to be resident beside the state pass)

struct GenParams {
  const float *partial, *W1, *b1, *W2, *b2;
  float *hidden, *w, *state;                          // state: the chunks' sum, in the layout of a partial
  const void *v, *q;                                  // q, o, status: prefix rows only
  __nv_bfloat16* o;
  const int* status;
  int B, H, R, P, ntok, nchunk, state_elems;
  int T;                                              // outputs per sample: C k k
  int group;                                          // samples per pass over the output layer (shared memory)
  int rows;                                           // of W2 per thread, 1 .. kRows
  int nhid, nred;                                     // blocks of the hidden layer per sample; blocks per head that sum the chunks
  int nmain;                                          // blocks of the output layer; the ones behind take prefix rows
  float inv_n, eps;
};

// Eight lanes' share of a 128-value stretch of a weight row: values 4 part + 32 i .. + 3 (kVec), part + 8 i (not kVec)
template <bool kVec>
__device__ __forceinline__ void load_row(float (&x)[16], const float* row, int n, int part, bool in) {
  if (kVec) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int c = 4 * part + 32 * i;
      const float4 y = in && c < n ? __ldg(reinterpret_cast<const float4*>(row + c)) : make_float4(0.f, 0.f, 0.f, 0.f);
      x[4 * i] = y.x; x[4 * i + 1] = y.y; x[4 * i + 2] = y.z; x[4 * i + 3] = y.w;
    }
  } else {
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      const int c = part + 8 * i;
      x[i] = in && c < n ? __ldg(row + c) : 0.f;
    }
  }
}
// acc[j][i] += row j's stretch (w[j]) . n values of sample min(first + i, last), for j < rows.  Several rows share a
// thread's loads of the samples' values: with one row at a time the shared-memory port was the limit.
template <bool kVec, int kRows, int kS>
__device__ __forceinline__ void dot_rows(float (&acc)[kRows][kS], const float (&w)[kRows][16], const float* y, size_t stride,
                                         int first, int last, int n, int part, int rows) {
  if (kVec) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int c = 4 * part + 32 * i;
      if (c < n) {
        float4 h[kS];
#pragma unroll
        for (int b = 0; b < kS; ++b) h[b] = *reinterpret_cast<const float4*>(y + min(first + b, last) * stride + c);
#pragma unroll
        for (int j = 0; j < kRows; ++j)
          if (j < rows) {
#pragma unroll
            for (int b = 0; b < kS; ++b)
              acc[j][b] = fmaf(w[j][4 * i], h[b].x, fmaf(w[j][4 * i + 1], h[b].y, fmaf(w[j][4 * i + 2], h[b].z, fmaf(w[j][4 * i + 3], h[b].w, acc[j][b]))));
          }
      }
    }
  } else {
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      const int c = part + 8 * i;
      if (c < n) {
#pragma unroll
        for (int b = 0; b < kS; ++b) {
          const float h = y[min(first + b, last) * stride + c];
#pragma unroll
          for (int j = 0; j < kRows; ++j) acc[j][b] = fmaf(w[j][i], h, acc[j][b]);
        }
      }
    }
  }
}
// Sums acc[0 .. kS) over eight neighbouring lanes, halving the samples that a lane still carries at each step
// (7 shuffles for 8 samples instead of 24): lane `part` returns the sum of sample part / (8 / kS).
template <int kS>
__device__ __forceinline__ float sum_lanes(float (&acc)[kS], int part) {
  int n = kS;
#pragma unroll
  for (int mask = 4; mask >= 1; mask >>= 1) {
    if (n > 1) {
      n >>= 1;
      const bool up = (part & mask) != 0;
#pragma unroll
      for (int i = 0; i < kS / 2; ++i)
        if (i < n) {
          const float send = up ? acc[i] : acc[i + n], keep = up ? acc[i + n] : acc[i];
          acc[i] = keep + __shfl_xor_sync(0xffffffffu, send, mask);
        }
    } else {
      acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], mask);
    }
  }
  return acc[0];
}
// o of the P prefix tokens of one (batch, head): relu(q) KV / (relu(q).z + eps), fp32 throughout
__device__ __forceinline__ void prefix_rows(const GenParams& p, int bh, float* smem) {
  float* qs = smem;                                   // [kGenPrefix][64]
  float* zs = qs + kGenPrefix * kD;                   // [64]
  float* red = zs + kD;                               // [kAGroups][kGenPrefix][64]
  constexpr int kPer = kD / kAGroups;                 // rows of KV per thread
  const int e = threadIdx.x & 63, ag = threadIdx.x >> 6;
  const size_t row0 = (size_t)bh * p.ntok;
  const int nchunk = p.nred ? 1 : p.nchunk;
  const __nv_bfloat16* q = (const __nv_bfloat16*)p.q + row0 * kD;
  for (int i = threadIdx.x; i < p.P * kD; i += kThreadsOut) qs[i] = fmaxf(__bfloat162float(q[i]), 0.f);
  griddep_wait();
  const bool gave_up = *reinterpret_cast<const volatile int*>(p.status) != 0;   // an earlier kernel gave up: o stays as it is
  const float* src = p.nred ? p.state + (size_t)bh * p.state_elems : p.partial + (size_t)bh * p.nchunk * p.state_elems;
  float kv[kPer], z = 0.f;
#pragma unroll
  for (int i = 0; i < kPer; ++i) kv[i] = 0.f;
  for (int c = 0; c < nchunk; ++c, src += p.state_elems) {            // in chunk order
#pragma unroll
    for (int i = 0; i < kPer; ++i) kv[i] += __ldcg(src + (kPer * ag + i) * kD + e);
    if (threadIdx.x < kD) z += __ldcg(src + kOffZ + threadIdx.x);
  }
  if (threadIdx.x < kD) zs[threadIdx.x] = z;
  __syncthreads();
  for (int t = 0; t < p.P; ++t) {
    float s = 0.f;
#pragma unroll
    for (int i = 0; i < kPer; ++i) s = fmaf(qs[t * kD + kPer * ag + i], kv[i], s);
    red[(ag * kGenPrefix + t) * kD + e] = s;
  }
  __syncthreads();
  for (int t = ag; t < p.P; t += kAGroups) {
    float den = p.eps;
#pragma unroll 16
    for (int a = 0; a < kD; ++a) den = fmaf(qs[t * kD + a], zs[a], den);
    float s = 0.f;
#pragma unroll
    for (int g = 0; g < kAGroups; ++g) s += red[(g * kGenPrefix + t) * kD + e];
    if (!gave_up) p.o[(row0 + t) * kD + e] = __float2bfloat16_rn(s / den);
  }
}

// One of the nred blocks that sum the chunks of head h of sample b
__device__ __forceinline__ void sum_chunks(const GenParams& p, int b, int h, int part) {
  constexpr int kVecs = (kD * kD + kD) / 4;           // KV and z
  griddep_wait();                                     // the state pass is complete
  const size_t bh = (size_t)b * p.H + h;
  const float4* src = reinterpret_cast<const float4*>(p.partial + bh * p.nchunk * p.state_elems);
  float4* dst = reinterpret_cast<float4*>(p.state + bh * p.state_elems);
  const int stride = p.state_elems / 4;
  for (int i = part * kThreads + threadIdx.x; i < kVecs; i += p.nred * kThreads) {
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int k0 = 0; k0 < p.nchunk; k0 += 8) {
      float4 x[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) x[k] = k0 + k < p.nchunk ? __ldcg(src + (size_t)(k0 + k) * stride + i) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int k = 0; k < 8; ++k) { s.x += x[k].x; s.y += x[k].y; s.z += x[k].z; s.w += x[k].w; }
    }
    dst[i] = s;
  }
}

// A block serves 8 values of r for one sample: per 1024 channels it forms the means in shared memory while the rows of
// W1 are already on their way, then warp w takes row r0 + w.
template <typename T, bool kVec>
__global__ void __launch_bounds__(kThreads, 2)
gen_hidden_kernel(const GenParams p) {
  __shared__ __align__(16) float mean[kTileC];
  griddep_launch_dependents();                        // (the grid behind this one waits for it before it reads hidden)
  if ((int)blockIdx.x >= p.nhid) {
    const int i = blockIdx.x - p.nhid;
    sum_chunks(p, blockIdx.y, i / p.nred, i % p.nred);
    return;
  }
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int r = blockIdx.x * 8 + warp, b = blockIdx.y, C = p.H * kD;
  const bool r_ok = r < p.R;
  const float* wrow = p.W1 + (size_t)(r_ok ? r : 0) * C;
  float dot = 0.f;
  for (int c0 = 0; c0 < C; c0 += kTileC) {
    float4 wv[kTileC / 128];                          // this lane's part of the row
#pragma unroll
    for (int i = 0; i < kTileC / 128; ++i) {
      const int c = c0 + 4 * lane + 128 * i;          // (C is a multiple of 64)
      const bool in = r_ok && c < C;
      if (kVec) wv[i] = in ? __ldg(reinterpret_cast<const float4*>(wrow + c)) : make_float4(0.f, 0.f, 0.f, 0.f);
      else wv[i] = in ? make_float4(__ldg(wrow + c), __ldg(wrow + c + 1), __ldg(wrow + c + 2), __ldg(wrow + c + 3)) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    if (c0 == 0) griddep_wait();                      // the state pass is complete
    __syncthreads();                                  // the previous tile's means have been consumed
    {
      constexpr int kPer = kTileC / kThreads;         // four channels per thread: all their loads in flight together
      const float* pv[kPer];
      float m[kPer];
      size_t row[kPer];
#pragma unroll
      for (int j = 0; j < kPer; ++j) {
        const int c = min(c0 + (int)threadIdx.x + kThreads * j, C - 1);
        const size_t bh = (size_t)b * p.H + c / kD;
        pv[j] = p.partial + bh * p.nchunk * p.state_elems + kOffVsum + c % kD;
        row[j] = bh * p.ntok * kD + c % kD;
        m[j] = 0.f;
      }
      for (int k0 = 0; k0 < p.nchunk; k0 += 4) {      // in chunk order
        float x[4][kPer];
#pragma unroll
        for (int k = 0; k < 4; ++k)
#pragma unroll
          for (int j = 0; j < kPer; ++j) x[k][j] = k0 + k < p.nchunk ? __ldcg(pv[j] + (size_t)(k0 + k) * p.state_elems) : 0.f;
#pragma unroll
        for (int k = 0; k < 4; ++k)
#pragma unroll
          for (int j = 0; j < kPer; ++j) m[j] += x[k][j];
      }
      // the v-sums run over all tokens; the pooling is over the grid: take the prefix rows out again
#pragma unroll 4
      for (int t = 0; t < p.P; ++t)
#pragma unroll
        for (int j = 0; j < kPer; ++j) m[j] -= to_f32(((const T*)p.v)[row[j] + (size_t)t * kD]);
#pragma unroll
      for (int j = 0; j < kPer; ++j) mean[threadIdx.x + kThreads * j] = m[j] * p.inv_n;   // (past C: weights of zero)
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < kTileC / 128; ++i) {
      const float4 sv = *reinterpret_cast<const float4*>(mean + 4 * lane + 128 * i);
      dot = fmaf(wv[i].x, sv.x, fmaf(wv[i].y, sv.y, fmaf(wv[i].z, sv.z, fmaf(wv[i].w, sv.w, dot))));
    }
  }
  dot = warp_sum(dot);
  if (lane == 0 && r_ok) {
    const float x = dot + (p.b1 ? p.b1[r] : 0.f);
    p.hidden[(size_t)b * p.R + r] = x / (1.f + expf(-x));
  }
}

// Eight lanes per row of W2, p.rows rows per thread, kS samples worked on together (their hidden vectors in shared memory).
// Two rows a thread share its loads of the hidden values; with four, fewer warps are left to hide the latencies with (32
// samples of 96 hidden units and 6912 outputs: 5.7 us in the loop over the samples against 4.0).
template <bool kVec, int kS>
__global__ void __launch_bounds__(kThreadsOut, 3)
gen_out_kernel(const GenParams p) {
  extern __shared__ __align__(16) float smem_g[];
  griddep_launch_dependents();                        // (the grid behind this one waits for it before it reads w or o)
  if ((int)blockIdx.x >= p.nmain) {
    prefix_rows(p, blockIdx.x - p.nmain, smem_g);
    return;
  }
  const int part = threadIdx.x & 7, sub = threadIdx.x >> 3, R = p.R;
  const int rows = p.rows, t0 = blockIdx.x * rows * kRowsPass, t_end = min(p.T, t0 + rows * kRowsPass);
  float w2[kRows][16], bias[kRows];
  auto load_w2 = [&](int r) {
#pragma unroll
    for (int j = 0; j < kRows; ++j) {
      const int t = t0 + kRowsPass * j + sub;
      load_row<kVec>(w2[j], p.W2 + (size_t)(t < t_end ? t : t0) * R + r, R - r, part, t < t_end);
    }
  };
  load_w2(0);
#pragma unroll
  for (int j = 0; j < kRows; ++j) {
    const int t = t0 + kRowsPass * j + sub;
    bias[j] = p.b2 && t < t_end ? __ldg(p.b2 + t) : 0.f;
  }
  griddep_wait();                                     // the hidden layer is complete
  for (int b0 = 0; b0 < p.B; b0 += p.group) {
    const int nb = min(p.group, p.B - b0);
    if (b0 > 0) __syncthreads();
    if (kVec) {
      for (int i = 4 * threadIdx.x; i < nb * R; i += 4 * kThreadsOut)
        *reinterpret_cast<float4*>(smem_g + i) = __ldcg(reinterpret_cast<const float4*>(p.hidden + (size_t)b0 * R + i));
    } else {
      for (int i = threadIdx.x; i < nb * R; i += kThreadsOut) smem_g[i] = __ldcg(p.hidden + (size_t)b0 * R + i);
    }
    __syncthreads();
    for (int bb = 0; bb < nb; bb += kS) {             // (a last group of samples is filled up with its last one)
      float acc[kRows][kS];
#pragma unroll
      for (int j = 0; j < kRows; ++j)
#pragma unroll
        for (int i = 0; i < kS; ++i) acc[j][i] = 0.f;
      for (int r = 0; r < R; r += 128) {
        if (r > 0 || (b0 + bb > 0 && R > 128)) load_w2(r);
        dot_rows<kVec>(acc, w2, smem_g + r, R, bb, nb - 1, R - r, part, rows);
      }
#pragma unroll
      for (int j = 0; j < kRows; ++j) {
        const float x = sum_lanes<kS>(acc[j], part);
        const int t = t0 + kRowsPass * j + sub, b = bb + part / (8 / kS);
        if (part % (8 / kS) == 0 && b < nb && t < t_end) p.w[(size_t)(b0 + b) * p.T + t] = x + bias[j];
      }
    }
  }
}

}  // namespace

cudaError_t dwc_static_kernels(const LinArgs& a, const LinPlan& p, const float** w, int* w_batch, cudaStream_t st) {
  const int T = a.s.H * kD * a.dwc->k * a.dwc->k;
  *w = (const float*)((char*)a.ws + p.off_kernel);
  *w_batch = T;
  if (a.dwc->R > 0) return cudaSuccess;
  *w_batch = 0;
  if (((uintptr_t)a.dwc->b2 & 15) == 0) {
    *w = a.dwc->b2;
    return cudaSuccess;
  }
  return cudaMemcpyAsync((char*)a.ws + p.off_kernel, a.dwc->b2, (size_t)T * sizeof(float), cudaMemcpyDeviceToDevice, st);
}

cudaError_t launch_sum_chunks(const LinArgs& a, const LinPlan& p, const float* partial, const float** state, cudaStream_t st) {
  GenParams g = {};
  g.partial = partial;
  g.state = (float*)((char*)a.ws + p.off_state);
  g.H = a.s.H;
  g.nchunk = p.nchunk;
  g.state_elems = p.state_elems;
  g.nred = 4;
  *state = g.state;
  return launch_programmatic(gen_hidden_kernel<__nv_bfloat16, true>, dim3(g.nred * a.s.H, a.s.B), kThreads, 0, st, g);
}

cudaError_t launch_dwc_generator_fast(const LinArgs& a, const LinPlan& p, const float* partial, bool prefix, const float** state,
                                      int* nchunk, cudaStream_t st) {
  const jv_shape& s = a.s;
  const jv_dwc& d = *a.dwc;
  // static kernels: a launch only for sums of enough chunks (its 3 us against the readers' round trips)
  const bool reduce = p.nchunk >= (d.R > 0 ? 3 : 8);
  *state = partial;
  *nchunk = p.nchunk;
  if (d.R == 0 && !prefix && !reduce) return cudaSuccess;
  GenParams g = {};
  g.state = (float*)((char*)a.ws + p.off_state);
  if (reduce) {
    g.nred = p.nchunk >= 8 ? 4 : 1;
    *state = g.state;
    *nchunk = 1;
  }
  g.partial = partial;
  g.W1 = d.W1;
  g.b1 = d.b1;
  g.W2 = d.W2;
  g.b2 = d.b2;
  g.hidden = (float*)((char*)a.ws + p.off_hidden);
  g.w = (float*)((char*)a.ws + p.off_kernel);
  g.v = a.v;
  g.q = a.q;
  g.o = (__nv_bfloat16*)a.o;
  g.B = s.B;
  g.H = s.H;
  g.R = d.R;
  g.P = s.P;
  g.ntok = shape_tokens(s);
  g.nchunk = p.nchunk;
  g.state_elems = p.state_elems;
  g.T = s.H * kD * d.k * d.k;
  g.inv_n = 1.f / (float)(s.Hg * s.Wg);               // pooling: the mean over the grid tokens
  g.eps = a.eps;
  const bool vec = d.R % 4 == 0 && (((uintptr_t)d.W1 | (uintptr_t)d.W2) & 15) == 0;
  size_t smem = 0;
  if (d.R > 0 || reduce) {
    g.nhid = ceil_div(d.R, 8);
    const dim3 grid(g.nhid + g.nred * s.H, s.B);
    const cudaError_t e = s.dtype == JV_F32 ? (vec ? launch_programmatic(gen_hidden_kernel<float, true>, grid, kThreads, 0, st, g)
                                                   : launch_programmatic(gen_hidden_kernel<float, false>, grid, kThreads, 0, st, g))
                                            : (vec ? launch_programmatic(gen_hidden_kernel<__nv_bfloat16, true>, grid, kThreads, 0, st, g)
                                                   : launch_programmatic(gen_hidden_kernel<__nv_bfloat16, false>, grid, kThreads, 0, st, g));
    if (e != cudaSuccess) return e;
  }
  if (d.R == 0 && !prefix) return cudaSuccess;
  if (d.R > 0) {
    size_t group = kMaxSmem / (d.R * sizeof(float));  // (R <= 1024: at least 12)
    group &= ~(size_t)7;
    g.group = (size_t)s.B < group ? s.B : (int)group;
    smem = (size_t)g.group * d.R * sizeof(float);
    g.rows = ceil_div(g.T, kRowsPass * device_sm_count());            // one wave of blocks
    if (g.rows > kRows) g.rows = kRows;
    g.nmain = ceil_div(g.T, g.rows * kRowsPass);
  }
  int blocks = g.nmain;
  if (prefix) {
    g.status = device_status_ptr();
    if (!g.status) return cudaErrorUnknown;
    blocks += s.B * s.H;
    const size_t need = (size_t)((1 + kAGroups) * kGenPrefix + 1) * kD * sizeof(float);
    if (smem < need) smem = need;
  }
  // one sample, two, four or eight at a time
  auto* out = !vec ? gen_out_kernel<false, 4> : s.B == 1 ? gen_out_kernel<true, 1> : s.B == 2 ? gen_out_kernel<true, 2>
              : s.B <= 4 ? gen_out_kernel<true, 4> : gen_out_kernel<true, 8>;
  return launch_programmatic(out, dim3(blocks), kThreadsOut, smem, st, g);
}

}  // namespace jv
