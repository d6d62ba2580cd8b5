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
  f32::layer_product<NT, TM, CPT, ST>(h1s, W1, st, w1, w2, acc);
  f32::layer_tanh<NT, TM, CPT>(h2s, b1, w2, acc);
  out_layer<NT, RM>(h2s, W2, b2, w2, w3, row0, M, Y);
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
    const cudaError_t e = cudaFuncSetAttribute(k_mlp3_f32<NT, TM, CPT, ST>,
                                               cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               C::floats(kMaxIn) * 4);
    if (e != cudaSuccess) return e;
    if (dev >= 0 && dev < 64) attr_set[dev] = true;
  }
  const float *W0 = params + sh.layer_offset(0), *W1 = params + sh.layer_offset(1),
              *W2 = params + sh.layer_offset(2);
  k_mlp3_f32<NT, TM, CPT, ST><<<(unsigned)((M + C::RM - 1) / C::RM), NT, smem, st>>>(
      X, ldr, ldc, W0, W0 + (size_t)sh.w[0] * sh.w[1], W1, W1 + (size_t)sh.w[1] * sh.w[2], W2,
      W2 + (size_t)sh.w[2] * sh.w[3], Y, M, sh.w[0], sh.w[1], sh.w[2], sh.w[3]);
  return cudaGetLastError();
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
  if (h <= 64) {
    if (per_sm <= 8) return run<128, 1, 4, 4>(X, ldr, ldc, params, p, Y, M, st);
    if (per_sm <= 16) return run<128, 2, 4, 4>(X, ldr, ldc, params, p, Y, M, st);
    return run<128, 4, 4, 4>(X, ldr, ldc, params, p, Y, M, st);
  }
  if (h <= 128) {
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
