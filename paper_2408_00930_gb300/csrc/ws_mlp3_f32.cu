// ws_mlp3_f32.cu -- the three-layer FP32 policy forward in one launch: the batched
// FP32 path's inference of the economy and the landscape (paper App. B: policy
// inference on the model held in global memory) and ws_policy_forward_noalloc.
//
// A CTA takes RM = 8 TM rows through all layers with the activations in shared memory
// (ws_mlp_f32.cuh); every output is k_dense_fp32's chain, equal bit for bit.  Three
// k_dense_fp32 launches passed each activation through memory and ran 16-deep stages
// with two barriers each: 300 rows of 16-128-128-20 51 us, 8,192 rows of 4-256-256-2
// 115 us, 8,192 rows of 24-256-256-48 116 us; here 10, 38 and
// 60 us (floors 4, 14 and 18: the FP32 pipe, for the first the chain of phases).
#include "ws_kernels.cuh"
#include "ws_mlp_f32.cuh"

namespace ws {

namespace {

constexpr int kMaxIn = 64;  // input widths
constexpr int kUnitIn = 24, kUnitOut = 48;  // k_mlp3_f32u's inputs and outputs

// NT threads, TM rows per thread group, CPT columns per thread (NPAD = NT / 8 CPT >=
// both hidden widths), ST stages of streamed weights.
template <int NT, int TM, int CPT, int ST>
struct MCfg {
  static constexpr int RM = 8 * TM, NPAD = NT / 8 * CPT;
  static constexpr bool kSmall = TM * CPT <= 16;  // separate h1 / h2 arrays
  static constexpr int HB = NPAD * RM;
  static constexpr int W_FLOATS = ST * f32::kKC * NPAD;
  // floats: [x, k4 x RM] [h1 (h2)] [h2] [weight stages]
  static int floats(int k4) { return k4 * RM + (kSmall ? 2 : 1) * HB + W_FLOATS; }
};

// The last layer: each of the NT / RM thread groups takes its share of the outputs,
// up to 12 at a time.
template <int NT, int RM>
__device__ __forceinline__ void out_layer(const float *H, const float *__restrict__ W,
                                          const float *__restrict__ b, int K, int N, long row0, int M,
                                          float *__restrict__ Y) {
  constexpr int G = NT / RM;
  auto put = [&](int r, int o, float v) {
    if (row0 + r < M) Y[(row0 + r) * N + o] = v;
  };
  for (int base = 0; base < N;) {
    const int left = N - base, per = (left + G - 1) / G;
    const float *Wb = W + base, *bb = b + base;
    auto put_b = [&](int r, int o, float v) { put(r, base + o, v); };
    if (per <= 1) {
      f32::layer_out<RM, 1>(H, Wb, bb, K, left, N, put_b);
      base = N;
    } else if (per <= 3) {
      f32::layer_out<RM, 3>(H, Wb, bb, K, left, N, put_b);
      base = N;
    } else if (per <= 4) {
      f32::layer_out<RM, 4>(H, Wb, bb, K, left, N, put_b);
      base = N;
    } else if (per <= 8) {
      f32::layer_out<RM, 8>(H, Wb, bb, K, left, N, put_b);
      base = N;
    } else {
      const int take = left < 12 * G ? left : 12 * G;
      f32::layer_out<RM, 12>(H, Wb, bb, K, take, N, put_b);
      base += take;
    }
  }
}

template <int NT, int TM, int CPT, int ST>
__global__ void __launch_bounds__(NT, NT == 256 ? 2 : 1)
    k_mlp3_f32(const float *__restrict__ X, long ldr, long ldc, const float *__restrict__ W0,
               const float *__restrict__ b0, const float *__restrict__ W1, const float *__restrict__ b1,
               const float *__restrict__ W2, const float *__restrict__ b2, float *__restrict__ Y, int M,
               int w0, int w1, int w2, int w3) {
  using C = MCfg<NT, TM, CPT, ST>;
  constexpr int RM = C::RM;
  extern __shared__ float4 smem4[];
  float *xs = (float *)smem4;
  const int k4 = (w0 + 3) & ~3, tid = threadIdx.x;
  float *h1s = xs + k4 * RM, *h2s = C::kSmall ? h1s + C::HB : h1s, *st = h2s + C::HB;
  const long row0 = (long)blockIdx.x * RM;
  if (ldc == 1) {  // row-major rows: walk k fastest
    for (int i = tid; i < RM * k4; i += NT) {
      const int k = i % k4, r = i / k4;
      xs[f32::act_idx<RM>(k, r)] = (row0 + r < M && k < w0) ? X[(row0 + r) * ldr + k] : 0.f;
    }
  } else {  // SoA: walk rows fastest
    for (int i = tid; i < RM * k4; i += NT) {
      const int r = i % RM, k = i / RM;
      xs[f32::act_idx<RM>(k, r)] =
          (row0 + r < M && k < w0) ? X[(row0 + r) * ldr + (long)k * ldc] : 0.f;
    }
  }
  __syncthreads();
  uint64_t acc[TM][CPT / 2];
  f32::layer_product<NT, TM, CPT, ST>(xs, W0, st, w0, w1, acc);
  f32::layer_tanh<NT, TM, CPT>(h1s, b0, w1, acc);
  f32::zero_pad<NT, C::RM>(h1s, w1);
  f32::layer_product<NT, TM, CPT, ST>(h1s, W1, st, w1, w2, acc);
  f32::layer_tanh<NT, TM, CPT>(h2s, b1, w2, acc);
  out_layer<NT, RM>(h2s, W2, b2, w2, w3, row0, M, Y);
}

// The output layer of k_mlp3_f32u's eight rows: thread (output, RPO rows).
template <int RPO, int P>
__device__ __forceinline__ void out_rows(const float *h2s, const float *w2s, const float *b2, float *Y,
                                         long row0, int M, int w2, int w3, int tid) {
  const int o = tid % w3, r0 = tid / w3 * RPO;
  if (r0 >= 8) return;
  const float b = __ldg(b2 + o);
  float acc[RPO];
#pragma unroll
  for (int r = 0; r < RPO; ++r) acc[r] = 0.f;
#pragma unroll 8
  for (int k = 0; k < w2; ++k) {
    const float w = w2s[k * w3 + o];
#pragma unroll
    for (int r = 0; r < RPO; ++r) acc[r] = fmaf(h2s[(r0 + r) * P + k], w, acc[r]);
  }
#pragma unroll
  for (int r = 0; r < RPO; ++r)
    if (row0 + r0 + r < M) Y[(row0 + r0 + r) * w3 + o] = acc[r] + b;
}

// Few rows, hidden widths up to HP = 64 or 128: eight rows per CTA and a thread per
// (unit, row group), as k_ctrl_f32u (ws_control_f32.cu).  With at most 16 rows per SM
// the time is one pass through the weights' latency and three dependent chains, not
// arithmetic: so all weights are asked for at once before the first product (the
// thread's W0 and W1 columns to registers, W2 to shared memory), where the tiled
// kernel's streamed stages took a barrier per eight reduction steps.  16-128-128-20,
// 1 / 300 / 2,400 rows: 11.3 / 12.3 / 14.4 us tiled, 8.3 / 10.3 / 12.3 us here;
// 4-64-64-2, 300 rows: 7.6 and 6.2 us.
template <int HP>
__global__ void __launch_bounds__(128)
    k_mlp3_f32u(const float *__restrict__ X, long ldr, long ldc, const float *__restrict__ W0,
                const float *__restrict__ b0, const float *__restrict__ W1, const float *__restrict__ b1,
                const float *__restrict__ W2, const float *__restrict__ b2, float *__restrict__ Y, int M,
                int w0, int w1, int w2, int w3) {
  constexpr int RM = 8, NT = 128, RPT = RM * HP / NT, P = HP + 4, XP = kUnitIn + 4;
  __shared__ __align__(16) float h1s[RM * P], h2s[RM * P], xs[RM * XP], w2s[HP * kUnitOut];
  const int tid = threadIdx.x, u = tid % HP, r0 = tid / HP * RPT;
  const long row0 = (long)blockIdx.x * RM;
  for (int i = tid; i < w2 * w3; i += NT)
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((uint32_t)__cvta_generic_to_shared(w2s + i)),
                 "l"(W2 + i) : "memory");
  float w1c[HP];
#pragma unroll
  for (int k = 0; k < HP; ++k) w1c[k] = (u < w2 && k < w1) ? __ldg(W1 + (size_t)k * w2 + u) : 0.f;
  float w0c[kUnitIn];
#pragma unroll
  for (int k = 0; k < kUnitIn; ++k) w0c[k] = (u < w1 && k < w0) ? __ldg(W0 + k * w1 + u) : 0.f;
  if (u >= w1)  // zeros past w1 (an infinite input times their zero weights is NaN)
    for (int r = 0; r < RPT; ++r) h1s[(r0 + r) * P + u] = 0.f;
  const float b0u = u < w1 ? __ldg(b0 + u) : 0.f, b1u = u < w2 ? __ldg(b1 + u) : 0.f;
  for (int i = tid; i < RM * w0; i += NT) {
    const int r = i / w0, k = i % w0;
    xs[r * XP + k] = row0 + r < M ? X[(row0 + r) * ldr + (long)k * ldc] : 0.f;
  }
  __syncthreads();
  {
    float z[RPT];
#pragma unroll
    for (int r = 0; r < RPT; ++r) z[r] = 0.f;
#pragma unroll
    for (int k = 0; k < kUnitIn; ++k)
      if (k < w0)
#pragma unroll
        for (int r = 0; r < RPT; ++r) z[r] = fmaf(xs[(r0 + r) * XP + k], w0c[k], z[r]);
#pragma unroll
    for (int r = 0; r < RPT; ++r) h1s[(r0 + r) * P + (u < w1 ? u : HP)] = tanhf(z[r] + b0u);
  }
  __syncthreads();
  {
    float acc[RPT];
#pragma unroll
    for (int r = 0; r < RPT; ++r) acc[r] = 0.f;
#pragma unroll
    for (int k4 = 0; k4 < HP; k4 += 4)
#pragma unroll
      for (int r = 0; r < RPT; ++r) {
        const float4 h = *(const float4 *)(h1s + (r0 + r) * P + k4);
        acc[r] = fmaf(h.x, w1c[k4], acc[r]);
        acc[r] = fmaf(h.y, w1c[k4 + 1], acc[r]);
        acc[r] = fmaf(h.z, w1c[k4 + 2], acc[r]);
        acc[r] = fmaf(h.w, w1c[k4 + 3], acc[r]);
      }
#pragma unroll
    for (int r = 0; r < RPT; ++r) h2s[(r0 + r) * P + u] = tanhf(acc[r] + b1u);
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();
  if (w3 <= NT / 8)
    out_rows<1, P>(h2s, w2s, b2, Y, row0, M, w2, w3, tid);
  else if (w3 <= NT / 4)
    out_rows<2, P>(h2s, w2s, b2, Y, row0, M, w2, w3, tid);
  else
    out_rows<4, P>(h2s, w2s, b2, Y, row0, M, w2, w3, tid);
}

template <int HP>
cudaError_t run_u(const float *X, long ldr, long ldc, const float *params, const PolicyShape &sh,
                  float *Y, int M, cudaStream_t st) {
  const float *W0 = params + sh.layer_offset(0), *W1 = params + sh.layer_offset(1),
              *W2 = params + sh.layer_offset(2);
  return launch_kernel(k_mlp3_f32u<HP>, dim3((unsigned)((M + 7) / 8)), dim3(128), 0, st, X, ldr, ldc, W0,
                       W0 + (size_t)sh.w[0] * sh.w[1], W1, W1 + (size_t)sh.w[1] * sh.w[2], W2,
                       W2 + (size_t)sh.w[2] * sh.w[3], Y, M, sh.w[0], sh.w[1], sh.w[2], sh.w[3]);
}

template <int NT, int TM, int CPT, int ST>
cudaError_t run(const float *X, long ldr, long ldc, const float *params, const PolicyShape &sh, float *Y,
                int M, cudaStream_t st) {
  using C = MCfg<NT, TM, CPT, ST>;
  const int smem = C::floats((sh.w[0] + 3) & ~3) * 4;
  // the shared-memory limit, once per device (idempotent, so a race on the flag is benign)
  static bool attr_set[64] = {};
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev < 0 || dev >= 64 || !attr_set[dev]) {
    const cudaError_t e = set_smem_limit(k_mlp3_f32<NT, TM, CPT, ST>, C::floats(kMaxIn) * 4);
    if (e != cudaSuccess) return e;
    if (dev >= 0 && dev < 64) attr_set[dev] = true;
  }
  const float *W0 = params + sh.layer_offset(0), *W1 = params + sh.layer_offset(1),
              *W2 = params + sh.layer_offset(2);
  return launch_kernel(k_mlp3_f32<NT, TM, CPT, ST>, dim3((unsigned)((M + C::RM - 1) / C::RM)), dim3(NT), smem,
                       st, X, ldr, ldc, W0, W0 + (size_t)sh.w[0] * sh.w[1], W1,
                       W1 + (size_t)sh.w[1] * sh.w[2], W2, W2 + (size_t)sh.w[2] * sh.w[3], Y, M, sh.w[0],
                       sh.w[1], sh.w[2], sh.w[3]);
}

}  // namespace

bool mlp3_f32_supported(const PolicyShape &p) {
  return p.w[0] <= kMaxIn && p.w[1] <= 256 && p.w[2] <= 256 && p.w[3] <= 128;
}

// The row tile by width and rows per SM, as the fused roll-out's (ws_control_f32.cu),
// whose products these are; weights are streamed for every tile here.
cudaError_t launch_mlp3_f32(const float *X, long ldr, long ldc, const float *params,
                            const PolicyShape &p, float *Y, int M, cudaStream_t st) {
  if (M <= 0) return cudaSuccess;
  const int h = p.w[1] > p.w[2] ? p.w[1] : p.w[2];
  int dev = 0, sms = 148;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int per_sm = (M + sms - 1) / sms;
  // 16 rows per SM: at 17 a third CTA per SM would wait for registers (206 x 128), and
  // the tiled kernel's two-tile wave is level (14.4 us for 2,433 rows of 16-128-128-20).
  // Wider inputs or outputs would not fit the registers and 48 KB of shared memory.
  const bool unit = per_sm <= 16 && p.w[0] <= kUnitIn && p.w[3] <= kUnitOut;
  if (h <= 64) {
    if (unit) return run_u<64>(X, ldr, ldc, params, p, Y, M, st);
    if (per_sm <= 8) return run<128, 1, 4, 4>(X, ldr, ldc, params, p, Y, M, st);
    if (per_sm <= 16) return run<128, 2, 4, 4>(X, ldr, ldc, params, p, Y, M, st);
    return run<128, 4, 4, 4>(X, ldr, ldc, params, p, Y, M, st);
  }
  if (h <= 128) {
    if (unit) return run_u<128>(X, ldr, ldc, params, p, Y, M, st);
    if (per_sm <= 8) return run<256, 1, 4, 4>(X, ldr, ldc, params, p, Y, M, st);
    if (per_sm <= 16) return run<256, 2, 4, 4>(X, ldr, ldc, params, p, Y, M, st);
    if (per_sm <= 200) return run<256, 4, 4, 4>(X, ldr, ldc, params, p, Y, M, st);
    return run<256, 8, 4, 3>(X, ldr, ldc, params, p, Y, M, st);
  }
  if (per_sm <= 8) return run<256, 1, 8, 4>(X, ldr, ldc, params, p, Y, M, st);
  if (per_sm <= 16) return run<256, 2, 8, 4>(X, ldr, ldc, params, p, Y, M, st);
  if (per_sm <= 32) return run<256, 4, 8, 4>(X, ldr, ldc, params, p, Y, M, st);
  return run<128, 8, 16, 2>(X, ldr, ldc, params, p, Y, M, st);
}

}  // namespace ws
