// ws_mlp_f32.cuh -- one row tile of a three-layer FP32 MLP on the CUDA cores,
// all layers in one CTA with the activations in shared memory.
//
// Shared by the fused FP32 roll-out kernel of the classic-control envs
// (ws_control_f32.cu) and the whole-MLP forward (ws_mlp3_f32.cu).  Every output
// element is the same chain as k_dense_fp32's: an FMA per input in k order from
// zero, then one add of the bias (and tanhf), so that the results are equal bit
// for bit and only the work split differs.
//
// NT threads take RM = 8 TM rows.  Thread (ty, tx), ty < 8 and tx < TX =
// NT / 8, of a wide layer owns rows ty TM .. + TM and columns 4 TX q + 4 tx .. + 4
// (CPT = NPAD / TX of them), two columns per packed fma.rn.f32x2.  Bound: the FP32 FMA
// pipe (128 per clock per SM; the packed form gives no more FMAs, but half the
// issue slots, which the shared-memory loads and the operand copies then use).
// At TM = 8, CPT = 16 a thread's k step is 64 packed FMAs against six 16-byte
// shared loads.  Activations lie [k][row] with the 4-row blocks of column k
// XOR-ed by k / 4, so that the writes of an epilogue (a thread holds consecutive
// columns), the k-th reads of the product and the row-wise reads of the narrow
// last layer are all free of bank conflicts without padding.
#pragma once

#include "ws_kernels.cuh"

namespace ws {
namespace f32 {

constexpr int kKC = 16;  // weight rows per stage of a streamed layer

// Asynchronous copy of BYTES (4 or 16) into shared memory, zeros if !valid.
template <int BYTES>
__device__ __forceinline__ void cp_async(void *dst, const void *src, bool valid) {
  const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
  if (BYTES == 16)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src),
                 "r"(valid ? 16 : 0)
                 : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(d), "l"(src),
                 "r"(valid ? 4 : 0)
                 : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Float index of (k, row) in an activation array of RM rows.
template <int RM>
__device__ __forceinline__ int act_idx(int k, int r) {
  return k * RM + ((((r >> 2) ^ ((k >> 2) & (RM / 4 - 1))) << 2) | (r & 3));
}

// Weight rows [k0, k0 + rows) of W[K][N] into st[rows][NPAD], zeros past K and N.
// vec: N and the base allow 16-byte copies.
template <int NT, int NPAD>
__device__ __forceinline__ void load_weights(float *st, const float *__restrict__ W, int k0, int rows,
                                             int K, int N, bool vec) {
  if (vec) {
    for (int i = threadIdx.x; i < rows * (NPAD / 4); i += NT) {
      const int k = i / (NPAD / 4), c = (i % (NPAD / 4)) * 4;
      const bool ok = k0 + k < K && c < N;
      cp_async<16>(st + k * NPAD + c, ok ? W + (size_t)(k0 + k) * N + c : W, ok);
    }
  } else {
    for (int i = threadIdx.x; i < rows * NPAD; i += NT) {
      const int k = i / NPAD, c = i % NPAD;
      const bool ok = k0 + k < K && c < N;
      cp_async<4>(st + k * NPAD + c, ok ? W + (size_t)(k0 + k) * N + c : W, ok);
    }
  }
}
__device__ __forceinline__ bool vec_weights(const float *W, int N) {
  return (N & 3) == 0 && ((uintptr_t)W & 15) == 0;
}

// Thread coordinates of the wide layers: a warp is 2 row groups x 16 column
// groups, so that a 16-byte load of the weights is two wavefronts for its 16
// distinct addresses and the activations' is one.
template <int NT>
__device__ __forceinline__ int tile_tx() {
  return (int)(threadIdx.x & 15) + (NT == 256 ? (int)(threadIdx.x >> 7) * 16 : 0);
}
template <int NT>
__device__ __forceinline__ int tile_ty() {
  return (int)(threadIdx.x >> 4) & 7;
}

// acc += A W over `rows` (a multiple of 4) weight rows in shared memory; the
// rows' activations start at column k0 of A.
template <int NT, int TM, int CPT>
__device__ __forceinline__ void mma_rows(const float *__restrict__ A, const float *__restrict__ Ws,
                                         int k0, int rows, uint64_t (&acc)[TM][CPT / 2]) {
  constexpr int RM = 8 * TM, TX = NT / 8, NPAD = TX * CPT;
  const int tx = tile_tx<NT>(), ty = tile_ty<NT>();
  const float *wp = Ws + tx * 4;
#pragma unroll(TM *CPT >= 64 ? 1 : 4)
  for (int k4 = 0; k4 < rows; k4 += 4) {
    const int f = ((k0 + k4) >> 2) & (RM / 4 - 1);
    const float *ap = A + (k0 + k4) * RM;
#pragma unroll
    for (int kk = 0; kk < 4; ++kk) {
      float a[TM];
      if (TM >= 4) {
#pragma unroll
        for (int q = 0; q < TM / 4; ++q) {
          const float4 v = *(const float4 *)(ap + kk * RM + (((ty * (TM / 4) + q) ^ f) << 2));
          a[4 * q] = v.x;
          a[4 * q + 1] = v.y;
          a[4 * q + 2] = v.z;
          a[4 * q + 3] = v.w;
        }
      } else if (TM == 2) {
        const float2 v = *(const float2 *)(ap + kk * RM + ((((ty >> 1) ^ f) << 2) | ((ty & 1) << 1)));
        a[0] = v.x;
        a[1] = v.y;
      } else {
        a[0] = ap[kk * RM + ((((ty >> 2) ^ f) << 2) | (ty & 3))];
      }
      uint64_t b[CPT / 2];
#pragma unroll
      for (int q = 0; q < CPT / 4; ++q) {
        const ulonglong2 v = *(const ulonglong2 *)(wp + (k4 + kk) * NPAD + 4 * TX * q);
        b[2 * q] = v.x;
        b[2 * q + 1] = v.y;
      }
#pragma unroll
      for (int i = 0; i < TM; ++i) {
        const uint64_t aa = f2_pack(a[i], a[i]);
#pragma unroll
        for (int j = 0; j < CPT / 2; ++j) acc[i][j] = f2_fma(aa, b[j], acc[i][j]);
      }
    }
  }
}

// A whole layer's product.  ST = 0: W lies in shared memory ([K rounded up to 4]
// [NPAD]); else it is streamed from global memory through ST stages of kKC rows
// in st, ST - 1 of them in flight (CTA barriers inside).
template <int NT, int TM, int CPT, int ST>
__device__ __forceinline__ void layer_product(const float *A, const float *W, float *st, int K, int N,
                                              uint64_t (&acc)[TM][CPT / 2]) {
  constexpr int NPAD = NT / 8 * CPT;
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < CPT / 2; ++j) acc[i][j] = 0ull;
  if (ST == 0) {
    mma_rows<NT, TM, CPT>(A, W, 0, (K + 3) & ~3, acc);
    return;
  }
  constexpr int S = ST > 0 ? ST : 1;
  const bool vec = vec_weights(W, N);
  const int nc = (K + kKC - 1) / kKC;
#pragma unroll
  for (int c = 0; c < S - 1; ++c) {
    if (c < nc) load_weights<NT, NPAD>(st + c * (kKC * NPAD), W, c * kKC, kKC, K, N, vec);
    cp_commit();
  }
  for (int c = 0; c < nc; ++c) {
    cp_wait<(S > 1 ? S - 2 : 0)>();
    __syncthreads();  // chunk c has landed for every thread; the stage of chunk c - 1 is free
    const int p = c + S - 1;
    if (p < nc) load_weights<NT, NPAD>(st + (p % S) * (kKC * NPAD), W, p * kKC, kKC, K, N, vec);
    cp_commit();
    mma_rows<NT, TM, CPT>(A, st + (c % S) * (kKC * NPAD), c * kKC, min(kKC, (K - c * kKC + 3) & ~3),
                          acc);
  }
  cp_wait<0>();
  __syncthreads();  // the stages are free
}

// tanh(acc + b) into H (columns past N are tanh(0) = 0, the next layer's zero padding;
// zero_pad where an input may be infinite, which times a zero weight is NaN).  Small
// tiles apply tanhf in registers; larger ones write the pre-activations and apply it in
// place over the array (the unrolled tanhf of 32 to 128 values per thread would not fit
// the instruction cache).  H may be the product's own input when the tile is large (a
// CTA barrier separates them).  Ends with a CTA barrier.
template <int NT, int TM, int CPT>
__device__ __forceinline__ void layer_tanh(float *H, const float *__restrict__ b, int N,
                                           const uint64_t (&acc)[TM][CPT / 2]) {
  constexpr int RM = 8 * TM, TX = NT / 8;
  constexpr bool kSmall = TM * CPT <= 16;
  const int tx = tile_tx<NT>(), ty = tile_ty<NT>();
  if (!kSmall) __syncthreads();  // every thread has read the product's input
#pragma unroll
  for (int q = 0; q < CPT / 4; ++q)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int col = 4 * TX * q + 4 * tx + j;
      const float bc = col < N ? __ldg(b + col) : 0.f;
      float z[TM];
#pragma unroll
      for (int i = 0; i < TM; ++i) {
        const float2 p = f2_unpack(acc[i][2 * q + (j >> 1)]);
        z[i] = ((j & 1) ? p.y : p.x) + bc;
        if (kSmall) z[i] = tanhf(z[i]);
      }
      float *o = H + col * RM;
      const int f = (col >> 2) & (RM / 4 - 1);
      if (TM >= 4) {
#pragma unroll
        for (int u = 0; u < TM / 4; ++u)
          *(float4 *)(o + (((ty * (TM / 4) + u) ^ f) << 2)) =
              make_float4(z[4 * u], z[4 * u + 1], z[4 * u + 2], z[4 * u + 3]);
      } else if (TM == 2) {
        *(float2 *)(o + ((((ty >> 1) ^ f) << 2) | ((ty & 1) << 1))) = make_float2(z[0], z[TM - 1]);
      } else {
        o[(((ty >> 2) ^ f) << 2) | (ty & 3)] = z[0];
      }
    }
  __syncthreads();
  if (!kSmall) {
    const int n4 = ((N + 3) & ~3) * (RM / 4);
#pragma unroll(NT == 256 ? 2 : 4)
    for (int i = threadIdx.x; i < n4; i += NT) {
      float4 v = ((float4 *)H)[i];
      v.x = tanhf(v.x);
      v.y = tanhf(v.y);
      v.z = tanhf(v.z);
      v.w = tanhf(v.w);
      ((float4 *)H)[i] = v;
    }
    __syncthreads();
  }
}

// Zeros in the columns from N to a multiple of 4, for every width that has such columns.
template <int NT, int RM>
__device__ __forceinline__ void zero_pad(float *H, int N) {
  if ((N & 3) == 0) return;
  const int n1 = N * (RM / 4), n4 = ((N + 3) & ~3) * (RM / 4);
  if ((int)threadIdx.x < n4 - n1) ((float4 *)H)[n1 + threadIdx.x] = make_float4(0.f, 0.f, 0.f, 0.f);
  __syncthreads();
}

// The narrow last layer: thread t takes row t % RM and the CO outputs from
// (t / RM) CO on of N (weight rows ld apart); put(row, output, value) receives the
// sum with its bias.
template <int RM, int CO, typename Put>
__device__ __forceinline__ void layer_out(const float *__restrict__ H, const float *__restrict__ W,
                                          const float *__restrict__ b, int K, int N, int ld, Put put) {
  const int r = threadIdx.x % RM, o0 = (int)(threadIdx.x / RM) * CO;
  if (o0 >= N) return;
  float acc[CO];
#pragma unroll
  for (int c = 0; c < CO; ++c) acc[c] = 0.f;
  const int r4 = r >> 2, rl = r & 3;
  int k = 0;
  // 16-byte weight loads where every row's share starts on 16 bytes and is whole
  const bool vec = CO % 4 == 0 && (ld & 3) == 0 && ((uintptr_t)W & 15) == 0 && o0 + CO <= N;
  if (vec) {
#pragma unroll 2
    for (; k + 4 <= K; k += 4) {
      const float *hp = H + k * RM + (((r4 ^ ((k >> 2) & (RM / 4 - 1))) << 2) | rl);
      const float *wp = W + k * ld + o0;
#pragma unroll
      for (int kk = 0; kk < 4; ++kk) {
        const float h = hp[kk * RM];
#pragma unroll
        for (int c = 0; c + 4 <= CO; c += 4) {
          const float4 w = *(const float4 *)(wp + kk * ld + c);
          acc[c] = fmaf(h, w.x, acc[c]);
          acc[c + 1] = fmaf(h, w.y, acc[c + 1]);
          acc[c + 2] = fmaf(h, w.z, acc[c + 2]);
          acc[c + 3] = fmaf(h, w.w, acc[c + 3]);
        }
      }
    }
  } else {
#pragma unroll(CO <= 3 ? 4 : 2)
    for (; k + 4 <= K; k += 4) {
      const float *hp = H + k * RM + (((r4 ^ ((k >> 2) & (RM / 4 - 1))) << 2) | rl);
      const float *wp = W + k * ld + o0;
#pragma unroll
      for (int kk = 0; kk < 4; ++kk) {
        const float h = hp[kk * RM];
#pragma unroll
        for (int c = 0; c < CO; ++c)
          if (c == 0 || o0 + c < N) acc[c] = fmaf(h, wp[kk * ld + c], acc[c]);
      }
    }
  }
  for (; k < K; ++k) {
    const float h = H[act_idx<RM>(k, r)];
#pragma unroll
    for (int c = 0; c < CO; ++c)
      if (c == 0 || o0 + c < N) acc[c] = fmaf(h, W[k * ld + o0 + c], acc[c]);
  }
#pragma unroll
  for (int c = 0; c < CO; ++c)
    if (o0 + c < N) put(r, o0 + c, acc[c] + b[o0 + c]);
}

}  // namespace f32
}  // namespace ws
