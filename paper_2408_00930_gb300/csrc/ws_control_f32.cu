// ws_control_f32.cu -- fused FP32 roll-out kernel of the classic-control envs
// (the control env and the acrobot, paper App. C): one launch runs a whole chunk
// of steps, each CTA keeping its row tile's env state and activations on chip.
//
// Paper grounding: Sec. 2 / App. B keep the env step, the policy forward, the
// sampling and the in-place store on the GPU; the envs are independent, so a
// tile's steps need nothing from outside the CTA.  The batched FP32 path ran six
// launches per step before (observe, three layers, draw, env step), each with its
// activations through global memory; the arithmetic here is theirs, operation by
// operation, so the records are equal bit for bit.
//
// A step is: layer 1 and 2 products with tanh (ws_mlp_f32.cuh), the two or three
// logits as one FMA chain each, then one thread per row draws the action, steps
// the env and writes the records.  W1, b3 and W3 stay in shared memory for the
// launch; W2 too up to 128 units (64 KB), else its rows are streamed from L2.
//
// What bounds it: the FP32 FMA pipe for many envs (131,072 envs, 4-256-256-2: 380
// us per step against 1,003 us for the six kernels; 67% of the pipe's cycles busy
// with the products' and tanhf's FMAs, floor 253 us), the step's own chain of
// dependent phases for few (1,000 envs, 4-64-64-2: 1.8 us per step against 32 us).
#include <math.h>

#include "ws_acrobot.cuh"
#include "ws_kernels.cuh"
#include "ws_mlp_f32.cuh"

namespace ws {

namespace {

struct FCart {
  static constexpr int OBS = 4, NA = 2;
};
struct FAcro {
  static constexpr int OBS = 6, NA = 3;
};
constexpr int kOP = 8;  // observation rows, padded to a multiple of 4 with zeros

// TM rows per thread group, CPT columns per thread (NPAD = NT / 8 CPT >= both
// hidden widths), ST: W2 resident (0) or streamed through ST stages.
template <typename E, int NT, int TM, int CPT, int ST>
struct Cfg {
  static constexpr int RM = 8 * TM, NPAD = NT / 8 * CPT;
  static constexpr bool kSmall = TM * CPT <= 16;  // separate h1 / h2 arrays
  static constexpr int S_X = 0;                            // [kOP][RM] observations
  static constexpr int S_H = S_X + kOP * RM;               // [NPAD][RM] h1 (then h2 in place)
  static constexpr int S_H2 = kSmall ? S_H + NPAD * RM : S_H;
  static constexpr int S_W1 = S_H2 + NPAD * RM;            // [kOP][NPAD]
  static constexpr int S_W2 = S_W1 + kOP * NPAD;           // resident W2, or two stages
  static constexpr int S_W3 = S_W2 + (ST == 0 ? NPAD * NPAD : ST * f32::kKC * NPAD);  // [NPAD][NA]
  static constexpr int S_LG = S_W3 + NPAD * E::NA + 4;     // [NA][RM] logits
  static constexpr int S_RN = S_LG + E::NA * RM;           // [7][RM] uniform, reset words, sin, cos
  static constexpr int FLOATS = S_RN + 7 * RM;
  static constexpr int SMEM = FLOATS * 4;
  static_assert(S_W1 % 4 == 0 && S_W2 % 4 == 0, "alignment");
  // the draws run on warps 2 and 3 beside the logits' chains where those leave them idle
  static constexpr bool kHelp = RM * E::NA <= 64 && 2 * RM <= 64;
};

template <typename E, int NT, int TM, int CPT, int ST>
__global__ void __launch_bounds__(NT, NT == 256 ? 2 : 1)
    k_ctrl_f32(Dev d, uint32_t off, uint32_t n_steps) {
  using C = Cfg<E, NT, TM, CPT, ST>;
  constexpr int OBS = E::OBS, NA = E::NA, RM = C::RM, NPAD = C::NPAD;
  constexpr bool ACRO = NA == 3;
  extern __shared__ float4 smem4[];
  float *sm = (float *)smem4;
  float *xs = sm + C::S_X, *h1s = sm + C::S_H, *h2s = sm + C::S_H2, *w1s = sm + C::S_W1;
  float *w2s = sm + C::S_W2, *w3s = sm + C::S_W3, *lg = sm + C::S_LG, *rn = sm + C::S_RN;
  const int tid = threadIdx.x;
  const int H0 = d.pol.w[1], H1 = d.pol.w[2];
  const float *W1 = d.params, *b1 = W1 + OBS * H0, *W2 = b1 + H0, *b2 = W2 + (size_t)H0 * H1,
              *W3 = b2 + H1, *b3 = W3 + H1 * NA;
  f32::load_weights<NT, NPAD>(w1s, W1, 0, kOP, OBS, H0, f32::vec_weights(W1, H0));
  if (ST == 0) f32::load_weights<NT, NPAD>(w2s, W2, 0, (H0 + 3) & ~3, H0, H1, f32::vec_weights(W2, H1));
  f32::cp_commit();
  for (int i = tid; i < H1 * NA; i += NT) w3s[i] = W3[i];
  for (int i = tid; i < kOP * RM; i += NT) xs[i] = 0.f;
  f32::cp_wait<0>();
  __syncthreads();  // the zeros of xs before the first observations

  const uint64_t k0 = d.k[0] + off;
  const uint32_t R = d.ring_steps, N = d.n_envs, S = d.n_slots;
  const bool lane = tid < RM;
  const uint32_t e0 = blockIdx.x * (uint32_t)RM, e = e0 + (uint32_t)tid;
  const bool valid = lane && e < N;
  float x = 0.f, v = 0.f, th = 0.f, w = 0.f;
  int tep = 0;
  if (valid) {
    x = d.s[e];
    v = d.s[N + e];
    th = d.s[2 * N + e];
    w = d.s[3 * N + e];
    tep = d.t[e];
  }
  // Philox words of step k for row q: the action uniform, or the reset words
  auto draw_action = [&](uint32_t k, int q) {
    rn[q] = u01(draw(d.seed, k, d.env_base + e0 + (uint32_t)q, 0, kTagAction, 0).x);
  };
  auto draw_reset = [&](uint32_t k, int q) {
    const uint4 r = draw(d.seed, k, d.env_base + e0 + (uint32_t)q, 0, kTagReset, 0);
    rn[RM + q] = __uint_as_float(r.x);
    rn[2 * RM + q] = __uint_as_float(r.y);
    rn[3 * RM + q] = __uint_as_float(r.z);
    rn[4 * RM + q] = __uint_as_float(r.w);
  };
  uint32_t row = (uint32_t)(k0 % R);
  for (uint32_t j = 0; j < n_steps; ++j) {
    const uint32_t k = (uint32_t)(k0 + j);
    // ---- observe
    float ob[OBS];
    if (lane) {
      if constexpr (ACRO) {
        sincosf(x, &ob[1], &ob[0]);
        sincosf(v, &ob[3], &ob[2]);
        ob[4] = th;
        ob[5] = w;
      } else {
        ob[0] = x;
        ob[1] = v;
        ob[2] = th;
        ob[3] = w;
      }
#pragma unroll
      for (int i = 0; i < OBS; ++i) xs[f32::act_idx<RM>(i, tid)] = ob[i];
    }
    __syncthreads();
    // ---- policy
    {
      uint64_t acc[TM][CPT / 2];
      f32::layer_product<NT, TM, CPT, 0>(xs, w1s, nullptr, OBS, H0, acc);
      f32::layer_tanh<NT, TM, CPT>(h1s, b1, H0, acc);
      f32::layer_product<NT, TM, CPT, ST>(h1s, ST == 0 ? w2s : W2, w2s, H0, H1, acc);
      f32::layer_tanh<NT, TM, CPT>(h2s, b2, H1, acc);
    }
    if (tid < RM * ((NA * RM + NT - 1) / NT > 1 ? NT / RM : NA)) {
      constexpr int CO = (NA * RM + NT - 1) / NT;
      f32::layer_out<RM, CO>(h2s, w3s, b3, H1, NA, NA, [&](int r, int o, float l) { lg[o * RM + r] = l; });
    }
    if (C::kHelp && tid >= 64) {
      const int h = tid - 64;
      if (h < RM) {
        draw_action(k, h);
        if constexpr (!ACRO) {
          const float a = xs[f32::act_idx<RM>(2, h)];
          rn[5 * RM + h] = sinf(a);
          rn[6 * RM + h] = cosf(a);
        }
      } else if (h < 2 * RM) {
        draw_reset(k, h - RM);
      }
    }
    __syncthreads();
    // ---- draw, env step, records
    if (lane) {
      if (!C::kHelp) {
        draw_action(k, tid);
        draw_reset(k, tid);
      }
      float l[NA];
#pragma unroll
      for (int c = 0; c < NA; ++c) l[c] = lg[c * RM + tid];
      float m = l[0];
#pragma unroll
      for (int c = 1; c < NA; ++c) m = fmaxf(m, l[c]);
      float ex[NA], Ssum = 0.f;
#pragma unroll
      for (int c = 0; c < NA; ++c) {
        ex[c] = expf(l[c] - m);
        Ssum += ex[c];
      }
      const float thr = rn[tid] * Ssum;
      float Cs = 0.f;
      int a = NA - 1;
      float la = l[NA - 1];
#pragma unroll
      for (int c = NA - 1; c >= 0; --c) {  // the first class whose running sum exceeds thr
        Cs = 0.f;
#pragma unroll
        for (int q = 0; q <= c; ++q) Cs += ex[q];
        if (thr < Cs) {
          a = c;
          la = l[c];
        }
      }
      float ns[4], rew;
      bool done;
      const int t2 = tep + 1;
      if constexpr (ACRO) {
        ns[0] = x;
        ns[1] = v;
        ns[2] = th;
        ns[3] = w;
        acro_step<false>(ns, (float)(a - 1), 0.2f);
        const bool term = acro_terminal<false>(ns);
        rew = term ? 0.0f : -1.0f;
        done = term || t2 >= (int)d.episode_limit;
      } else {
        const float sn = C::kHelp ? rn[5 * RM + tid] : sinf(th);
        const float cs = C::kHelp ? rn[6 * RM + tid] : cosf(th);
        const float u = a ? 10.0f : -10.0f;
        const float xacc = u - 0.5f * x - 0.1f * v;
        const float thacc = 9.8f * sn - 0.3f * cs * u;
        ns[0] = x + 0.02f * v;
        ns[1] = v + 0.02f * xacc;
        ns[2] = th + 0.02f * w;
        ns[3] = w + 0.02f * thacc;
        rew = 1.0f;
        done = fabsf(ns[0]) > 2.4f || fabsf(ns[2]) > 0.21f || t2 >= (int)d.episode_limit;
      }
      if (valid) {
        const size_t o = (size_t)row * S + e;
        float *obr = d.r_obs + (size_t)row * OBS * S + e;
#pragma unroll
        for (int i = 0; i < OBS; ++i) obr[(size_t)i * S] = ob[i];
        ((int32_t *)d.r_act)[o] = a;
        d.r_logp[o] = (la - m) - logf(Ssum);
        d.r_rew[o] = rew;
        d.r_done[o] = (uint8_t)done;
        if (d.r_pout) {
          float *po = d.r_pout + (size_t)row * NA * S + e;
#pragma unroll
          for (int c = 0; c < NA; ++c) po[(size_t)c * S] = l[c];
        }
        if (j + 1 == n_steps) {
#pragma unroll
          for (int c = 0; c < NA; ++c) d.out[(size_t)e * NA + c] = l[c];
        }
      }
      if (done) {
        const float lim = ACRO ? 0.1f : 0.05f;
        x = uniform(__float_as_uint(rn[RM + tid]), -lim, lim);
        v = uniform(__float_as_uint(rn[2 * RM + tid]), -lim, lim);
        th = uniform(__float_as_uint(rn[3 * RM + tid]), -lim, lim);
        w = uniform(__float_as_uint(rn[4 * RM + tid]), -lim, lim);
        tep = 0;
      } else {
        x = ns[0];
        v = ns[1];
        th = ns[2];
        w = ns[3];
        tep = t2;
      }
    }
    row = (row + 1 == R) ? 0 : row + 1;
  }
  if (valid) {
    d.s[e] = x;
    d.s[N + e] = v;
    d.s[2 * N + e] = th;
    d.s[3 * N + e] = w;
    d.t[e] = tep;
  }
}

template <typename E, int NT, int TM, int CPT, int ST>
cudaError_t run(const Dev &d, uint32_t off, uint32_t n, cudaStream_t st) {
  using C = Cfg<E, NT, TM, CPT, ST>;
  cudaError_t e = cudaFuncSetAttribute(k_ctrl_f32<E, NT, TM, CPT, ST>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM);
  if (e != cudaSuccess) return e;
  k_ctrl_f32<E, NT, TM, CPT, ST>
      <<<(d.n_envs + C::RM - 1) / C::RM, NT, C::SMEM, st>>>(d, off, n);
  return cudaGetLastError();
}

// The tile by hidden width and env count (us per step of the control env on 152
// SMs, rows per CTA 8 / 16 / 32 / 64).  While tiles of RM rows leave SMs without a
// CTA, a smaller tile shortens the step's chain; past that the larger tile has the
// better FMA-to-load ratio, until its last wave is too ragged.
//   width 64    1,000 envs: 1.82 1.91 2.21 3.96   5,000: 5.4 3.4 3.2 4.0   131,072: 104 57 35.3 35.9
//   width 128   1,000 envs: 4.1 4.3 5.2 8.8   20,000: 57 32 22.6 23.4   131,072: 362 188 119 105
//   width 256   1,000 envs: 18.7 19.7 23.3 34.5   5,000: 72 47 36 34.5   131,072: 1472 752 473 380
template <typename E>
cudaError_t run_env(const Dev &d, uint32_t off, uint32_t n, cudaStream_t st) {
  const int h = d.pol.w[1] > d.pol.w[2] ? d.pol.w[1] : d.pol.w[2];
  int dev = 0, sms = 148;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const uint32_t per_sm = (d.n_envs + (uint32_t)sms - 1) / (uint32_t)sms;
  if (h <= 64) {
    if (per_sm <= 8) return run<E, 128, 1, 4, 0>(d, off, n, st);
    if (per_sm <= 16) return run<E, 128, 2, 4, 0>(d, off, n, st);
    return run<E, 128, 4, 4, 0>(d, off, n, st);
  }
  if (h <= 128) {
    if (per_sm <= 8) return run<E, 256, 1, 4, 0>(d, off, n, st);
    if (per_sm <= 16) return run<E, 256, 2, 4, 0>(d, off, n, st);
    if (per_sm <= 200) return run<E, 256, 4, 4, 0>(d, off, n, st);
    return run<E, 256, 8, 4, 0>(d, off, n, st);
  }
  if (per_sm <= 8) return run<E, 256, 1, 8, 4>(d, off, n, st);
  if (per_sm <= 16) return run<E, 256, 2, 8, 4>(d, off, n, st);
  if (per_sm <= 32) return run<E, 256, 4, 8, 4>(d, off, n, st);
  return run<E, 128, 8, 16, 2>(d, off, n, st);
}

}  // namespace

bool control_f32_supported(const PolicyShape &sh) {
  const bool cart = sh.w[0] == FCart::OBS && sh.w[3] == FCart::NA;
  const bool acro = sh.w[0] == FAcro::OBS && sh.w[3] == FAcro::NA;
  return (cart || acro) && sh.w[1] <= 256 && sh.w[2] <= 256;
}

cudaError_t launch_control_f32(const Dev &d, uint32_t off, uint32_t n_steps, cudaStream_t st) {
  if (d.pol.w[3] == FAcro::NA) return run_env<FAcro>(d, off, n_steps, st);
  return run_env<FCart>(d, off, n_steps, st);
}

}  // namespace ws
