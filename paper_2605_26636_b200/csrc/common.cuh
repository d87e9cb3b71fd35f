// Shared host/device helpers of libjetvit (internal; not part of the C ABI).
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>
#include <utility>

#include "jetvit.h"

namespace jv {

// ---- device status word ---------------------------------------------------
// One int per device lives in api.cu; kernels receive its device address and OR
// error bits into it.  Bit 0: a bounded wait ran out.
constexpr int kStatusTimeout = 1;

int* device_status_ptr();        // device address of the status word (nullptr on failure)
void count_launch(int n = 1);    // launch counter behind jv_launch_count()

// ---- per-device facts --------------------------------------------------------
// The library may be used on several GPUs from one process (one device current per
// call), so whatever CUDA keeps per device is cached per device here.
constexpr int kMaxDevices = 64;
constexpr int kDefaultSmCount = 148;   // B200; used for planning when no device can be asked
int current_device();            // index of the current device, -1 if it cannot be read
int device_sm_count();           // SM count of the current device (kDefaultSmCount without one)

// Runs `f` (which returns a cudaError_t) once per device, with that device current:
// the opt-in to more than 48 KB of dynamic shared memory is a per-device function
// attribute.  Two host threads may both run f; it is idempotent.
class OncePerDevice {
 public:
  template <typename F>
  cudaError_t run(F f) {
    const int d = current_device();
    if (d < 0 || d >= kMaxDevices) return f();
    if (done_[d].load(std::memory_order_acquire)) return cudaSuccess;
    const cudaError_t e = f();
    if (e == cudaSuccess) done_[d].store(1, std::memory_order_release);
    return e;
  }

 private:
  std::atomic<int> done_[kMaxDevices] = {};
};

// ---- programmatic launches ----------------------------------------------------
// Every kernel of the tensor-core and fp32 paths is launched with programmatic stream serialisation: it may start, and do
// what depends on nothing (barriers, tensor memory, first loads of weights), while the launch ahead of it drains, which takes
// 2 to 4 us off every boundary between two launches.  The rules:
//   - a kernel waits (griddep_wait) before it reads what an earlier launch may have written and before it writes anything;
//     a launch is then complete only after the one ahead of it, so completion is transitive along the stream;
//   - it lets the next launch go (griddep_launch_dependents) only after its tensor memory is allocated (the next one's
//     allocation would otherwise wait for memory that this one could never get), and, where the next one reads the call's
//     inputs before its own wait, only after its own wait: whoever produced them is complete then.
__device__ __forceinline__ void griddep_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void griddep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

template <typename... Params, typename... Args>
cudaError_t launch_cluster(bool programmatic, void (*kernel)(Params...), int cluster, dim3 grid, int threads, size_t smem, cudaStream_t st,
                           Args&&... args) {
  // a grid of clusters of `cluster` blocks along x; 0: no clusters.  (A kernel that copies between shared memories of a cluster
  // needs the attribute for a cluster of one, too.)
  cudaLaunchAttribute attr[2];
  int n = 0;
  if (programmatic) {
    attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[n++].val.programmaticStreamSerializationAllowed = 1;
  }
  if (cluster > 0) {
    attr[n].id = cudaLaunchAttributeClusterDimension;
    attr[n].val.clusterDim.x = cluster;
    attr[n].val.clusterDim.y = 1;
    attr[n++].val.clusterDim.z = 1;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = attr;
  cfg.numAttrs = n;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
  count_launch();
  return e;
}
template <typename... Params, typename... Args>
cudaError_t launch_programmatic(void (*kernel)(Params...), dim3 grid, int threads, size_t smem, cudaStream_t st, Args&&... args) {
  return launch_cluster(true, kernel, 0, grid, threads, smem, st, std::forward<Args>(args)...);
}

// ---- element access -------------------------------------------------------
__device__ __forceinline__ float to_f32(float x) { return x; }
__device__ __forceinline__ float to_f32(__nv_bfloat16 x) { return __bfloat162float(x); }
__device__ __forceinline__ void from_f32(float* p, float x) { *p = x; }
__device__ __forceinline__ void from_f32(__nv_bfloat16* p, float x) { *p = __float2bfloat16_rn(x); }

__device__ __forceinline__ float warp_max(float x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x = fmaxf(x, __shfl_xor_sync(0xffffffffu, x, o));
  return x;
}
__device__ __forceinline__ float warp_sum(float x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  return x;
}

static inline int ceil_div(int a, int b) { return (a + b - 1) / b; }
// tokens per (batch, head): prefix tokens, then the grid
static inline int shape_tokens(const jv_shape& s) { return s.P + s.Hg * s.Wg; }
static inline size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

// Element strides of the inputs q, k, v over (token, head, batch); o is always [B, H, N, D] contiguous.
struct InStrides {
  int64_t tok, head, batch;
};
static inline InStrides in_strides(const jv_shape& s) {
  const int64_t n = shape_tokens(s);
  if (s.in_layout == JV_LAYOUT_BNHD) {
    const int64_t ts = s.in_tok_stride ? s.in_tok_stride : (int64_t)s.H * s.D;
    return InStrides{ts, (int64_t)s.D, n * ts};
  }
  return InStrides{(int64_t)s.D, n * s.D, (int64_t)s.H * n * s.D};
}
static inline bool in_strided(const jv_shape& s) { return s.in_layout != JV_LAYOUT_BHND; }

// ---- plan of the linear-attention workspace --------------------------------
// State per (batch, head): (D+1) x (D+1) fp32, S[a][e] = sum_j pk[j][a] * pv[j][e]
// with pk = [relu(k) | 1], pv = [v | 1]:  S[a<D][e<D] = KV, S[a][D] = z (k-sum),
// S[D][e] = v-sum, S[D][D] = N.
struct LinPlan {
  int D1;            // D + 1
  int state_elems;   // D1 * D1 rounded up to a multiple of 4
  int chunk_tokens;  // tokens per phase-1 chunk
  int nchunk;        // chunks per (batch, head)
  size_t off_partial, off_state, off_hidden, off_kernel, total;  // byte offsets into ws
  // token-wise dynamic convolution on the tensor-core path: bf16 copies of W1, W2, the hidden layer
  // [B, ntok, R] and the kernels of all tokens as planes [B, C*k*k/64, ntok, 64] (bf16)
  size_t off_tok_w1, off_tok_w2, off_tok_hidden, off_tok_kernel;
};
LinPlan lin_plan(const jv_shape& s, const jv_dwc* dwc);

// ---- kernels' host launchers (each returns a cudaError_t from the launch) ---
struct AttnArgs {
  const void *q, *k, *v;
  void* o;
  int BH, Hg, Wg, D;
  int H;           // heads: (batch, head) index bh = b * H + h
  InStrides in;    // element strides of q, k, v (the tensor-core paths honour them; the others need the default)
  bool strided;    // in differs from the contiguous [B, H, N, D] strides
  int P;       // prefix tokens in front of the Hg x Wg grid tokens (full attention: folded into the "grid")
  int wh, ww;  // window size (wh >= Hg and ww >= Wg: one window = full attention)
  float scale;
  int dtype;
};
cudaError_t launch_attn_generic(const AttnArgs& a, cudaStream_t st, bool windows_only = false);
// the P prefix queries of window attention on their own, ahead of the launch of the windows, which leaves `free_sms` SMs
// to it (bf16, D == 64, contiguous)
cudaError_t launch_attn_prefix(const AttnArgs& a, int free_sms, const int* status, cudaStream_t st);
// fp32 tensors at D == 64: register-tiled fp32 kernel (full and windowed attention, prefix tokens)
bool attn_f32_supported(const AttnArgs& a);
cudaError_t launch_attn_f32(const AttnArgs& a, cudaStream_t st);
// on the tensor cores, fp32 values as sums of three bf16 terms, six of their nine products, sums in fp32 (without the prefix queries, whose launch
// it overlaps if that is the one ahead)
cudaError_t launch_attn_f32_tc(const AttnArgs& a, bool overlap, int* status, cudaStream_t st);
// tcgen05 path: bf16, D == 64.  full = true: F over all N tokens; else W with (wh, ww)
// windows whose width ww is a power of two <= 128 (a tile is a box of ww x 128/ww tokens).
bool attn_tc_supported(const AttnArgs& a, bool full);
int attn_tc_ctas(const AttnArgs& a, bool full);   // CTAs (one per SM) of its launch
cudaError_t launch_attn_tc(const AttnArgs& a, bool full, int* status, cudaStream_t st);
// tcgen05 path for windows of one or two 128-token tiles (bf16, D == 64, at most 16 prefix tokens): two windows per CTA
bool attn_w4_supported(const AttnArgs& a);
int attn_w4_ctas(const AttnArgs& a);   // CTAs (one per SM) of its launch
cudaError_t launch_attn_w4(const AttnArgs& a, int* status, cudaStream_t st);
// tcgen05 path at head_dim 128 (bf16, N >= 128, no prefix tokens in W): two query tiles per CTA.
// full = true: F over all N tokens; else W with windows whose width is a power of two <= 128
bool attn_d128_supported(const AttnArgs& a, bool full);
cudaError_t launch_attn_d128(const AttnArgs& a, bool full, int* status, cudaStream_t st);
// tcgen05 path for full attention (bf16, D == 64), one query tile per CTA with its keys over four slots: all of a call, or what is left of
// it behind whole rounds of the four-tile kernel, by the cost of either
bool attn_split_supported(const AttnArgs& a);
cudaError_t launch_attn_split(const AttnArgs& a, int* status, cudaStream_t st);
// tcgen05 path for full attention (bf16, D == 64): four query tiles per CTA
bool attn_f4_supported(const AttnArgs& a);
// whole_groups > 0: only that many groups of four query tiles, of the floor(tiles / 4) whole ones of every head, head by head
cudaError_t launch_attn_f4(const AttnArgs& a, int* status, cudaStream_t st, int whole_groups = 0);
// time of a call on this kernel or the two-tile one, whichever is shorter, in rounds of items of four query tiles
float attn_f4_cost(int ntiles, int BH);

struct LinArgs {
  const void *q, *k, *v;
  void* o;
  jv_shape s;
  float eps;
  const jv_dwc* dwc;  // host struct holding device pointers, or nullptr
  void* ws;
};
cudaError_t launch_linear_generic(const LinArgs& a, const LinPlan& p, cudaStream_t st);
bool linear_fast_supported(const LinArgs& a);
cudaError_t launch_linear_fast(const LinArgs& a, const LinPlan& p, cudaStream_t st);
// bf16 tensors at D == 128 without the convolution
bool linear_d128_supported(const LinArgs& a);
cudaError_t launch_linear_d128(const LinArgs& a, const LinPlan& p, cudaStream_t st);
// fp32 tensors at D == 64, no convolution or 3 x 3 kernels (pooled or static)
bool linear_f32_supported(const LinArgs& a);
cudaError_t launch_linear_f32(const LinArgs& a, const LinPlan& p, cudaStream_t st);
// the kernel generator at D == 64, launched behind the grid that wrote the chunk partials (layout of lin_common.cuh); a grid
// launched with programmatic serialisation behind it that waits for it finds the kernels and everything before them
// complete.  prefix: the rows of o of the P <= kGenPrefix prefix tokens, too (bf16).  *state, *nchunk: where such a grid finds
// the heads' states, and in how many partials each.
constexpr int kGenPrefix = 16;
cudaError_t launch_dwc_generator_fast(const LinArgs& a, const LinPlan& p, const float* partial, bool prefix, const float** state,
                                      int* nchunk, cudaStream_t st);
// the chunk partials of every head summed in chunk order (what the generator does beside its hidden layer) by a launch of its own
cudaError_t launch_sum_chunks(const LinArgs& a, const LinPlan& p, const float* partial, const float** state, cudaStream_t st);
// where the convolution kernels of a call are: generated ones in ws + off_kernel, static ones in place; *w_batch: floats
// from sample to sample.  To be called ahead of the state pass (static kernels off 16 bytes are copied into ws).
cudaError_t dwc_static_kernels(const LinArgs& a, const LinPlan& p, const float** w, int* w_batch, cudaStream_t st);
// bf16, D == 64, 3 x 3 kernels: the apply pass with the convolution fused in
bool linear_conv_supported(const LinArgs& a);
cudaError_t launch_linear_apply_conv(const LinArgs& a, const LinPlan& p, const float* partial, int nchunk, const float* w,
                                     int w_batch, int* status, cudaStream_t st);
// shared by both linear paths: hidden = SiLU(W1 s + b1), w = W2 hidden + b2, with
// s = vsum / N read from vsum[bh * bh_stride + e]
cudaError_t launch_dwc_generator(const LinArgs& a, const LinPlan& p, const float* vsum, int bh_stride,
                                 cudaStream_t st);

// Focused feature map of Eq. 3 over every token row of q and k -> qf, kf (same shape and type)
cudaError_t launch_focus_map(const void* q, const void* k, void* qf, void* kf, const jv_shape& s, float p, cudaStream_t st);

// Token-wise dynamic convolution (Table 1): o (which holds the attention output) += the convolution
// of V with every grid token's own kernels.  Generic: everything per token on the fly, any type.
cudaError_t launch_dwc_tokenwise_generic(const LinArgs& a, cudaStream_t st);
// bf16, head_dim 64, 3 x 3, R a multiple of 64: generator as two tensor-core GEMMs, then the convolution
bool dwc_tokenwise_fast_supported(const LinArgs& a);
cudaError_t launch_dwc_tokenwise_fast(const LinArgs& a, const LinPlan& p, int* status, cudaStream_t st);
// the projection GEMM kernel on its own terms: D = act(A W^T + bias), bf16, fp32 accumulation.
//   planes_in:  A is [B, a_planes, N, 64] (K block kb = plane kb % a_planes), else A is [B, N, 64 * kblocks]
//   planes_out: D is [B, F / 64, N, 64] (feature block fb = plane fb), else D is [B, N, F]
//   W: [F, 64 * kblocks], bias fp32 [F] or null, silu: apply x / (1 + exp(-x)) to the result;
//   f16_in: A and W hold fp16 instead of bf16; f16_out: D is stored as fp16 instead of bf16
cudaError_t launch_proj_gemm(bool planes_in, bool planes_out, const void* A, const void* W, const float* bias, void* D, int B,
                             int N, int kblocks, int a_planes, int F, bool silu, bool f16_in, bool f16_out, int* status,
                             cudaStream_t st);

// Projections either side of a mixer (bf16, D == 64): qkv = true computes q, k, v (d0, d1, d2)
// from x [B, N, C]; qkv = false computes y (d0) [B, N, C] from x = o [B, H, N, 64].
bool proj_tc_available();
cudaError_t launch_proj_tc(bool qkv, const void* x, const void* w, const float* bias, void* d0, void* d1, void* d2,
                           const jv_shape& s, int* status, cudaStream_t st);

}  // namespace jv
