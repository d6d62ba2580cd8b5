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
// What bounds it: the FP32 FMA pipe for many envs (131,072 envs, 4-256-256-2: 372
// us per step against 1,003 us for the six kernels; 67% of the pipe's cycles busy
// with the products' and tanhf's FMAs, floor 253 us; at 255 registers the 64-row tile
// spills 32 bytes), the step's own chain of dependent phases for few (1,000 envs, 4-64-64-2: 1.2 us per step against 32 us).
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

// State of a row's env.
struct Row {
  float x = 0.f, v = 0.f, th = 0.f, w = 0.f;  // acrobot: (th1, th2, w1, w2)
  int tep = 0;
};
__device__ __forceinline__ void row_load(const Dev &d, Row &s, uint32_t e) {
  const uint32_t N = d.n_envs;
  s.x = d.s[e];
  s.v = d.s[N + e];
  s.th = d.s[2 * N + e];
  s.w = d.s[3 * N + e];
  s.tep = d.t[e];
}
__device__ __forceinline__ void row_store(const Dev &d, const Row &s, uint32_t e) {
  const uint32_t N = d.n_envs;
  d.s[e] = s.x;
  d.s[N + e] = s.v;
  d.s[2 * N + e] = s.th;
  d.s[3 * N + e] = s.w;
  d.t[e] = s.tep;
}
template <typename E>
__device__ __forceinline__ void row_observe(const Row &s, float (&ob)[E::OBS]) {
  if constexpr (E::NA == 3) {
    sincosf(s.x, &ob[1], &ob[0]);
    sincosf(s.v, &ob[3], &ob[2]);
    ob[4] = s.th;
    ob[5] = s.w;
  } else {
    ob[0] = s.x;
    ob[1] = s.v;
    ob[2] = s.th;
    ob[3] = s.w;
  }
}
// The draw from the logits l, the env step (sn, cs of the pole angle), the records and
// the auto-reset; rp[0] the action uniform, rp[rs], rp[2 rs], ... the reset words.
template <typename E>
__device__ __forceinline__ void row_step(const Dev &d, Row &s, const float (&ob)[E::OBS],
                                         const float (&l)[E::NA], const float *rp, int rs, float sn,
                                         float cs, bool valid, uint32_t e, uint32_t row, bool last) {
  constexpr int OBS = E::OBS, NA = E::NA;
  constexpr bool ACRO = NA == 3;
  const uint32_t S = d.n_slots;
  float m = l[0];
#pragma unroll
  for (int c = 1; c < NA; ++c) m = fmaxf(m, l[c]);
  float ex[NA], Ssum = 0.f;
#pragma unroll
  for (int c = 0; c < NA; ++c) {
    ex[c] = expf(l[c] - m);
    Ssum += ex[c];
  }
  const float thr = rp[0] * Ssum;
  int a = NA - 1;
  float la = l[NA - 1];
#pragma unroll
  for (int c = NA - 1; c >= 0; --c) {  // the first class whose running sum exceeds thr
    float Cs = 0.f;
#pragma unroll
    for (int q = 0; q <= c; ++q) Cs += ex[q];
    if (thr < Cs) {
      a = c;
      la = l[c];
    }
  }
  float ns[4], rew;
  bool done;
  const int t2 = s.tep + 1;
  if constexpr (ACRO) {
    ns[0] = s.x;
    ns[1] = s.v;
    ns[2] = s.th;
    ns[3] = s.w;
    acro_step<false>(ns, (float)(a - 1), 0.2f);
    const bool term = acro_terminal<false>(ns);
    rew = term ? 0.0f : -1.0f;
    done = term || t2 >= (int)d.episode_limit;
  } else {
    const float u = a ? 10.0f : -10.0f;
    const float xacc = u - 0.5f * s.x - 0.1f * s.v;
    const float thacc = 9.8f * sn - 0.3f * cs * u;
    ns[0] = s.x + 0.02f * s.v;
    ns[1] = s.v + 0.02f * xacc;
    ns[2] = s.th + 0.02f * s.w;
    ns[3] = s.w + 0.02f * thacc;
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
    if (last) {
#pragma unroll
      for (int c = 0; c < NA; ++c) d.out[(size_t)e * NA + c] = l[c];
    }
  }
  if (done) {
    const float lim = ACRO ? 0.1f : 0.05f;
    s.x = uniform(__float_as_uint(rp[rs]), -lim, lim);
    s.v = uniform(__float_as_uint(rp[2 * rs]), -lim, lim);
    s.th = uniform(__float_as_uint(rp[3 * rs]), -lim, lim);
    s.w = uniform(__float_as_uint(rp[4 * rs]), -lim, lim);
    s.tep = 0;
  } else {
    s.x = ns[0];
    s.v = ns[1];
    s.th = ns[2];
    s.w = ns[3];
    s.tep = t2;
  }
}

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
  static constexpr int S_W2 = S_W1 + kOP * NPAD;           // resident W2, or ST stages
  static constexpr int S_W3 = S_W2 + (ST == 0 ? NPAD * NPAD : ST * f32::kKC * NPAD);  // [NPAD][NA]
  static constexpr int S_LG = S_W3 + NPAD * E::NA + 4;     // [NA][RM] logits
  static constexpr int S_RN = S_LG + E::NA * RM;           // [7][RM] uniform, reset words, sin, cos
  static constexpr int FLOATS = S_RN + 7 * RM;
  static constexpr int SMEM = FLOATS * 4;
  static_assert(S_W1 % 4 == 0 && S_W2 % 4 == 0, "alignment");
  // the draws run on warps 2 and 3 beside the logits' chains where those leave them idle
  static constexpr bool kHelp = RM * E::NA <= 64 && 2 * RM <= 64;
};

// PAD: H0 is no multiple of 4 (in the kernel of the other widths the test alone costs 3%
// at 256 units: 391 against 378 us per step).
template <typename E, int NT, int TM, int CPT, int ST, bool PAD>
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
  const uint32_t R = d.ring_steps, N = d.n_envs;
  const bool lane = tid < RM;
  const uint32_t e0 = blockIdx.x * (uint32_t)RM, e = e0 + (uint32_t)tid;
  const bool valid = lane && e < N;
  Row s;
  if (valid) row_load(d, s, e);
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
      row_observe<E>(s, ob);
#pragma unroll
      for (int i = 0; i < OBS; ++i) xs[f32::act_idx<RM>(i, tid)] = ob[i];
    }
    __syncthreads();
    // ---- policy
    {
      uint64_t acc[TM][CPT / 2];
      f32::layer_product<NT, TM, CPT, 0>(xs, w1s, nullptr, OBS, H0, acc);
      f32::layer_tanh<NT, TM, CPT>(h1s, b1, H0, acc);
      if (PAD) f32::zero_pad<NT, RM>(h1s, H0);
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
      const float sn = ACRO ? 0.f : C::kHelp ? rn[5 * RM + tid] : sinf(s.th);
      const float cs = ACRO ? 0.f : C::kHelp ? rn[6 * RM + tid] : cosf(s.th);
      row_step<E>(d, s, ob, l, rn + tid, RM, sn, cs, valid, e, row, j + 1 == n_steps);
    }
    row = (row + 1 == R) ? 0 : row + 1;
  }
  if (valid) row_store(d, s, e);
}

// ------------------------------------------------------------ unit per thread
// Hidden widths up to HP = 64 or 128: eight rows per CTA, thread (unit, row group) with
// its W1 and W2 columns in registers, so that layer 2 is one 16-byte broadcast of h1
// per four FMAs and the step's chain is the FMA chains themselves.  (In the tiled
// kernel the weights come from shared memory for every two rows: 25 cycles per k at
// 64 units, 41 at 128, against 4 for the dependent FMA.)  Warp 0 takes the logits and
// the rows' steps, warp 2 the next step's draws, warp 3 sin and cos of the pole angle.
template <typename E, int HP>
struct Uc {
  static constexpr int RM = 8, NT = 128, RPT = RM * HP / NT;  // rows per thread
  static constexpr int P = HP + 4;                            // row stride of h1, h2
  static constexpr int W3P = HP + 4;
  static constexpr int FLOATS = 2 * RM * P + E::NA * W3P + RM * 8 + E::NA * RM + 12 * RM;
};

template <typename E, int HP>
__global__ void __launch_bounds__(128, HP == 64 ? 4 : 2)
    k_ctrl_f32u(Dev d, uint32_t off, uint32_t n_steps) {
  using C = Uc<E, HP>;
  constexpr int OBS = E::OBS, NA = E::NA, RM = C::RM, RPT = C::RPT;
  constexpr bool ACRO = NA == 3;
  __shared__ __align__(16) float sm[C::FLOATS];
  float *h1s = sm, *h2s = h1s + RM * C::P, *w3s = h2s + RM * C::P;  // [row][unit], W3 [out][unit]
  float *xs = w3s + NA * C::W3P;                                    // [row][8] observations
  float *lg = xs + RM * 8, *rn = lg + NA * RM, *sc = rn + 10 * RM;
  const int tid = threadIdx.x, u = tid % HP, g = tid / HP, r0 = g * RPT;
  const int H0 = d.pol.w[1], H1 = d.pol.w[2];
  const float *W1 = d.params, *b1 = W1 + OBS * H0, *W2 = b1 + H0, *b2 = W2 + (size_t)H0 * H1,
              *W3 = b2 + H1, *b3 = W3 + H1 * NA;
  // this unit's columns; zeros past the widths
  float w1c[OBS], w2c[HP];
#pragma unroll
  for (int k = 0; k < OBS; ++k) w1c[k] = u < H0 ? __ldg(W1 + k * H0 + u) : 0.f;
#pragma unroll
  for (int k = 0; k < HP; ++k) w2c[k] = (u < H1 && k < H0) ? __ldg(W2 + (size_t)k * H1 + u) : 0.f;
  const float b1u = u < H0 ? __ldg(b1 + u) : 0.f, b2u = u < H1 ? __ldg(b2 + u) : 0.f;
  for (int i = tid; i < NA * HP; i += C::NT) {
    const int o = i / HP, k = i % HP;
    w3s[o * C::W3P + k] = k < H1 ? __ldg(W3 + k * NA + o) : 0.f;
  }
  const uint64_t k0 = d.k[0] + off;
  const uint32_t R = d.ring_steps;
  const bool lane = tid < RM;
  const uint32_t e0 = blockIdx.x * (uint32_t)RM, e = e0 + (uint32_t)tid;
  const bool valid = lane && e < d.n_envs;
  Row s;
  if (valid) row_load(d, s, e);
  // step k's Philox words into buffer p: row q's action uniform (q < RM) or row q -
  // RM's reset words, one instruction stream for both
  auto draws = [&](uint32_t k, int q, int p) {
    const bool act = q < RM;
    const int qr = act ? q : q - RM;
    const uint4 r = draw(d.seed, k, d.env_base + e0 + (uint32_t)qr, 0, act ? kTagAction : kTagReset, 0);
    float *o = rn + p * 5 * RM + qr;
    if (act) {
      o[0] = u01(r.x);
    } else {
      o[RM] = __uint_as_float(r.x);
      o[2 * RM] = __uint_as_float(r.y);
      o[3 * RM] = __uint_as_float(r.z);
      o[4 * RM] = __uint_as_float(r.w);
    }
  };
  if (tid >= 64 && tid < 64 + 2 * RM) draws((uint32_t)k0, tid - 64, 0);
  // units past H0 keep zeros (an infinite observation times their zero weights is NaN):
  // their results go to the column past the units
  const int uc = u < H0 ? u : HP;
  if (u >= H0)
    for (int r = 0; r < RPT; ++r) h1s[(r0 + r) * C::P + u] = 0.f;
  uint32_t row = (uint32_t)(k0 % R);
  for (uint32_t j = 0; j < n_steps; ++j) {
    const uint32_t k = (uint32_t)(k0 + j);
    const int par = (int)(j & 1u);
    float ob[OBS];
    if (lane) {
      row_observe<E>(s, ob);
#pragma unroll
      for (int i = 0; i < OBS; ++i) xs[tid * 8 + i] = ob[i];
    }
    __syncthreads();
    // ---- layer 1 of this unit for its rows
#pragma unroll
    for (int r = 0; r < RPT; ++r) {
      float z = 0.f;
#pragma unroll
      for (int i = 0; i < OBS; ++i) z = fmaf(xs[(r0 + r) * 8 + i], w1c[i], z);
      h1s[(r0 + r) * C::P + uc] = tanhf(z + b1u);
    }
    __syncthreads();
    // ---- layer 2
    {
      float acc[RPT];
#pragma unroll
      for (int r = 0; r < RPT; ++r) acc[r] = 0.f;
#pragma unroll
      for (int k4 = 0; k4 < HP; k4 += 4)
#pragma unroll
        for (int r = 0; r < RPT; ++r) {
          const float4 h = *(const float4 *)(h1s + (r0 + r) * C::P + k4);
          acc[r] = fmaf(h.x, w2c[k4], acc[r]);
          acc[r] = fmaf(h.y, w2c[k4 + 1], acc[r]);
          acc[r] = fmaf(h.z, w2c[k4 + 2], acc[r]);
          acc[r] = fmaf(h.w, w2c[k4 + 3], acc[r]);
        }
#pragma unroll
      for (int r = 0; r < RPT; ++r) h2s[(r0 + r) * C::P + u] = tanhf(acc[r] + b2u);
    }
    __syncthreads();
    // ---- logits (warp 0), beside the next draws (warp 2) and sin / cos (warp 3)
    if (tid < RM * NA) {
      const int r = tid % RM, o = tid / RM;
      float acc = 0.f;
#pragma unroll
      for (int k4 = 0; k4 < HP; k4 += 4) {  // (zero products past H1 leave the sum as it is)
        const float4 h = *(const float4 *)(h2s + r * C::P + k4);
        const float4 w = *(const float4 *)(w3s + o * C::W3P + k4);
        acc = fmaf(h.x, w.x, acc);
        acc = fmaf(h.y, w.y, acc);
        acc = fmaf(h.z, w.z, acc);
        acc = fmaf(h.w, w.w, acc);
      }
      lg[o * RM + r] = acc + b3[o];
    }
    if (tid >= 64 && tid < 64 + 2 * RM) draws(k + 1, tid - 64, par ^ 1);
    if (!ACRO) {
      if (tid >= 96) {
        if (tid < 96 + RM) {
          const float a = xs[(tid - 96) * 8 + 2];
          sc[tid - 96] = sinf(a);
          sc[RM + tid - 96] = cosf(a);
        }
        __syncwarp();
        asm volatile("bar.arrive 1, 64;" ::: "memory");
      } else if (tid < 32) {
        asm volatile("bar.sync 1, 64;" ::: "memory");
      }
    }
    if (tid < 32) {
      __syncwarp();
      if (lane) {
        float l[NA];
#pragma unroll
        for (int c = 0; c < NA; ++c) l[c] = lg[c * RM + tid];
        row_step<E>(d, s, ob, l, rn + par * 5 * RM + tid, RM, ACRO ? 0.f : sc[tid],
                    ACRO ? 0.f : sc[RM + tid], valid, e, row, j + 1 == n_steps);
      }
    }
    row = (row + 1 == R) ? 0 : row + 1;
  }
  if (valid) row_store(d, s, e);
}

template <typename E, int HP>
cudaError_t run_u(const Dev &d, uint32_t off, uint32_t n, cudaStream_t st) {
  k_ctrl_f32u<E, HP><<<(d.n_envs + 7) / 8, 128, 0, st>>>(d, off, n);
  return cudaGetLastError();
}

template <typename E, int NT, int TM, int CPT, int ST>
cudaError_t run(const Dev &d, uint32_t off, uint32_t n, cudaStream_t st) {
  using C = Cfg<E, NT, TM, CPT, ST>;
  const auto kernel = (d.pol.w[1] & 3) ? k_ctrl_f32<E, NT, TM, CPT, ST, true>
                                       : k_ctrl_f32<E, NT, TM, CPT, ST, false>;
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM);
  if (e != cudaSuccess) return e;
  kernel<<<(d.n_envs + C::RM - 1) / C::RM, NT, C::SMEM, st>>>(d, off, n);
  return cudaGetLastError();
}

// The kernel and tile by hidden width and env count (us per step of the control env on
// 152 SMs; "unit" is k_ctrl_f32u, numbers are rows per tiled CTA).  While tiles of RM
// rows leave SMs without a CTA, a smaller tile shortens the step's chain; past that the
// larger tile has the better FMA-to-load ratio, until its last wave is too ragged.
//   width 64    1,000 envs: unit 1.23, 32 2.21   2,432: unit 1.46, 32 2.27   5,000: unit 3.11,
//               32 3.2, 64 4.0   131,072: unit 53, 32 35.3, 64 35.9
//   width 128   1,000 envs: unit 2.89, 32 5.2   2,432: unit 3.61, 32 5.3   20,000: unit 29.6,
//               32 22.6, 64 23.4   131,072: unit 186, 32 119, 64 105
//   width 256   1,000 envs: 8 17.3, 16 19.7, 32 23.3, 64 34.5   5,000: 72 47 36 33.3
//               131,072: 1,472 752 473 372
template <typename E>
cudaError_t run_env(const Dev &d, uint32_t off, uint32_t n, cudaStream_t st) {
  const int h = d.pol.w[1] > d.pol.w[2] ? d.pol.w[1] : d.pol.w[2];
  int dev = 0, sms = 148;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const uint32_t per_sm = (d.n_envs + (uint32_t)sms - 1) / (uint32_t)sms;
  if (h <= 64) {
    if (per_sm <= 16) return run_u<E, 64>(d, off, n, st);
    return run<E, 128, 4, 4, 0>(d, off, n, st);
  }
  if (h <= 128) {
    if (per_sm <= 16) return run_u<E, 128>(d, off, n, st);
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
