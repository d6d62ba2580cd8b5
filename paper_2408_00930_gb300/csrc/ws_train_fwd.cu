// ws_train_fwd.cu -- fused forward pass of the actor-critic update: gather, both
// hidden layers and the output layer of a policy and its critic in one launch.
//
// Paper grounding: Sec. 2 and App. B feed the trainer in place from the roll-out
// store; a row here is a recorded (step, slot) of the ring.
//
// Per 128-row tile: layer 1 in FP32 FMAs (k in order from zero, then the bias),
// tanhf, h1 written for the backward pass and split into BF16 hi + lo operand
// tiles; layer 2 as three tcgen05 products per K step (as k_gemm_tc); tanhf, h2
// written; the output layer in FP32 FMAs.  The parts ran as a gather, a thin GEMM,
// a 128 x 128-tile GEMM that read h1 twice, and a thin output layer (65,536 rows x
// 4-256-256-2: 20 + 63 + 17 us per network with a 64 MB activation read between each);
// here 58,368 rows of both networks take 87 us: issue slots 53% busy, the 60 M tanhf (two
// SFU results each, 7.3 per clock per SM measured) 27 us, tensor pipe 21%; the rest are
// the phases' loads and tails (long scoreboard) that the second CTA does not cover.
#include <math.h>

#include "ws_train_tc.cuh"

namespace ws {

namespace {

using namespace ttc;

struct Net {
  const float *W1, *b1, *b2, *W3, *b3;
  const uint8_t *image;  // packed W2
  float *h1, *h2, *out;
};
struct Nets {
  Net n[2];
  int count;
};

template <int H>
struct FwdSmem {
  using G = Geo<H>;
  static constexpr int OFF_B = (G::REG + 1023) / 1024 * 1024;
  static constexpr int OFF_BAR = OFF_B + G::B_BYTES;
  static constexpr int OFF_X = OFF_BAR + ((int)sizeof(Bars) + 15) / 16 * 16;
  // after the observations: W1, b1, b2 and W3 of the network in work, where they fit
  static int off_w(int xp) { return OFF_X + kRows * xp * 4; }
  static int w_floats(int in, int out) { return (in + 2 + out) * H; }
  static bool w_fits(int in, int xp, int out) {
    return off_w(xp) + w_floats(in, out) * 4 + 1024 <= kSmemPerCta;
  }
  static int bytes(int in, int xp, int out) {
    return off_w(xp) + (w_fits(in, xp, out) ? w_floats(in, out) * 4 : 0) + 1024;
  }
};

// W2[k][n] (FP32, row-major) as the MMA's B operand, hi and lo per K = 16 chunk:
// core matrices of 8 rows x 16 bytes, K-adjacent ones 128 bytes apart.  back: the
// data gradient's operand, B[n][k] = W2[n][k].
template <int H>
__global__ void k_pack_w2(const float *__restrict__ W2a, const float *__restrict__ W2c,
                          uint8_t *__restrict__ img, size_t stride, int back) {
  using G = Geo<H>;
  const float *W2 = blockIdx.y ? W2c : W2a;
  uint8_t *o = img + blockIdx.y * stride;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < H * H; i += gridDim.x * blockDim.x) {
    const int a = i / H, b = i % H;
    const int n = back ? a : b, k = back ? b : a;
    const float v = W2[i];
    const uint32_t hi = tc::pack_bf16x2(v, 0.f), lo = tc::pack_bf16x2(v - tc::bf16_lo(hi), 0.f);
    const size_t p = (size_t)(k / 16) * G::CHUNK + (size_t)(n >> 3) * 256 + ((k & 15) >> 3) * 128 +
                     (n & 7) * 16 + (k & 7) * 2;
    *(uint16_t *)(o + p) = (uint16_t)hi;
    *(uint16_t *)(o + p + H * 32) = (uint16_t)lo;
  }
}

// Output layer over one staged pass: thread (row, g) sums units g CTW / 2 .. of the
// pass into acc (FP32 FMAs in unit order).
template <int H, int OUT>
__device__ __forceinline__ void out_pass(const float *ct, const float *__restrict__ W3, int c0,
                                         float (&acc)[OUT]) {
  using G = Geo<H>;
  const int r = threadIdx.x & 127, g = threadIdx.x >> 7;
  constexpr int L = G::CTW / (kCT / kRows);
  const float *h = ct + r * G::CP + g * L;
  const float4 *w = (const float4 *)(W3 + (size_t)(c0 + g * L) * OUT);  // 16-byte aligned: c0 + g L is a multiple of 16
#pragma unroll(OUT <= 3 ? 4 : 1)
  for (int k = 0; k < L; k += 4) {
    const float4 hv = *(const float4 *)(h + k);
    float wv[4 * OUT];
#pragma unroll
    for (int q = 0; q < OUT; ++q) {
      const float4 v = w[(k / 4) * OUT + q];
      wv[4 * q] = v.x;
      wv[4 * q + 1] = v.y;
      wv[4 * q + 2] = v.z;
      wv[4 * q + 3] = v.w;
    }
#pragma unroll
    for (int o = 0; o < OUT; ++o) {
      acc[o] = fmaf(hv.x, wv[o], acc[o]);
      acc[o] = fmaf(hv.y, wv[OUT + o], acc[o]);
      acc[o] = fmaf(hv.z, wv[2 * OUT + o], acc[o]);
      acc[o] = fmaf(hv.w, wv[3 * OUT + o], acc[o]);
    }
  }
}

// One tile of one network by the compute warps (OUT = 0: no output layer here).
// Returns false if the accumulator's wait ran out.
template <int H, int OUT, int XV>
__device__ __forceinline__ bool fwd_tile(const Net &net, Bars *bars, uint8_t *reg, float *xs, int in,
                                         int xp, int tile, uint32_t tmem, uint32_t ph_acc,
                                         uint32_t &ph_af, const Dev &d, const Rows &rw, int next) {
  using G = Geo<H>;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int l16 = lane & 15, rh = lane >> 4;
  const uint32_t a = tc::smem_u32(reg);
  const size_t row0 = (size_t)tile * kRows;
  // ---- layer 1, one 64-unit K block at a time
  bool okw = true;
#pragma unroll 1
  for (int kb = 0; kb < G::KB; ++kb) {
    const int col = kb * 64 + l16 * 4;
    const float4 b = *(const float4 *)(net.b1 + col);
#pragma unroll 1
    for (int i0 = 0; i0 < kWR16; i0 += 8) {  // eight rows at a time
      float z[4][4];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) z[i][j] = 0.f;
      const float *xr = xs + (warp * kWR16 + i0 + rh) * xp;
#pragma unroll 4
      for (int k = 0; k < in; ++k) {
        const float4 w = *(const float4 *)(net.W1 + k * H + col);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float x = xr[2 * i * xp + k];
          z[i][0] = fmaf(x, w.x, z[i][0]);
          z[i][1] = fmaf(x, w.y, z[i][1]);
          z[i][2] = fmaf(x, w.z, z[i][2]);
          z[i][3] = fmaf(x, w.w, z[i][3]);
        }
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        z[i][0] = tanhf(z[i][0] + b.x);
        z[i][1] = tanhf(z[i][1] + b.y);
        z[i][2] = tanhf(z[i][2] + b.z);
        z[i][3] = tanhf(z[i][3] + b.w);
      }
      if (i0 == 0) okw = wait_block(bars, kb, ph_af) && okw;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int r = warp * kWR16 + i0 + 2 * i + rh;
        *(float4 *)(net.h1 + (row0 + r) * H + col) = make_float4(z[i][0], z[i][1], z[i][2], z[i][3]);
        store_a(a, r, l16 * 4, z[i]);
      }
    }
    tc::fence_async_smem();
    tc::fence_before_sync();
    __syncwarp();
    if (lane == 0) arrive(&bars->a);
  }
  float xn[XV];
  if (next >= 0) load_x<true>(d, rw, next, in, xn);
  // ---- layer 2's accumulator, then tanh and the output layer
  const bool ok = call(tc::mbar_wait(&bars->acc, ph_acc, tc::kDrainNs) && okw);
  if (!ok) return false;
  tc::fence_after_sync();
  float *ct = (float *)reg;  // the operand tiles are free: every product has completed
  float acc[OUT > 0 ? OUT : 1];
#pragma unroll
  for (int o = 0; o < OUT; ++o) acc[o] = 0.f;
#pragma unroll 1
  for (int c0 = 0; c0 < H; c0 += G::CTW) {
    if (c0) csync();  // the last pass's output sums have read ct
    stage_acc<H>(tmem, ct, c0, warp, lane);
    tc::fence_before_sync();
    csync();
    constexpr int LPR = G::CTW / 4, RPW = 32 / LPR;  // lanes per row, rows per warp access
    const int c = (lane % LPR) * 4;
    const float4 b = *(const float4 *)(net.b2 + c0 + c);
#pragma unroll 2
    for (int i = 0; i < kWR16; i += RPW) {
      const int r = warp * kWR16 + i + lane / LPR;
      float4 v = *(float4 *)(ct + r * G::CP + c);
      v.x = tanhf(v.x + b.x);
      v.y = tanhf(v.y + b.y);
      v.z = tanhf(v.z + b.z);
      v.w = tanhf(v.w + b.w);
      *(float4 *)(net.h2 + (row0 + r) * H + c0 + c) = v;
      if (OUT > 0) *(float4 *)(ct + r * G::CP + c) = v;
    }
    if (OUT > 0) {
      csync();
      out_pass<H, (OUT > 0 ? OUT : 1)>(ct, net.W3, c0, acc);
    }
  }
  if (next >= 0) store_x(xn, xp, xs);
  csync();  // ct is free
  if (OUT > 0) {
    // the two unit groups' sums of a row
    float *sp = ct;  // [2][128][OUT]
#pragma unroll
    for (int o = 0; o < OUT; ++o) sp[tid * OUT + o] = acc[o];
    csync();
    for (int i = tid; i < kRows * OUT; i += kCT) {
      constexpr int P = kRows * (OUT > 0 ? OUT : 1);
      net.out[row0 * OUT + i] = (sp[i] + sp[P + i]) + __ldg(net.b3 + i % (OUT > 0 ? OUT : 1));
    }
    csync();
  }
  return true;
}

template <int H, int OUT, int XV>
__global__ void __launch_bounds__(kThreads, 2)
    k_train_fwd(Dev d, Rows rw, int in, int xp, int off_w, const __grid_constant__ Nets nets) {
  using G = Geo<H>;
  using S = FwdSmem<H>;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = tc::smem_u32(smem_raw);
  uint8_t *sm = smem_raw + ((1024u - (raw & 1023u)) & 1023u);
  Bars *bars = (Bars *)(sm + S::OFF_BAR);
  float *xs = (float *)(sm + S::OFF_X);
  float *ws = off_w ? (float *)(sm + off_w) : nullptr;
  const int tid = threadIdx.x, warp = tid >> 5;
  if (tid == 0) bars_init(bars);
  if (warp == kCW) tc::tmem_alloc(&bars->tmem, H);
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = bars->tmem;
  const int tiles = (int)((rw.rows + kRows - 1) / kRows);
  bool ok = true;
  if (warp == kCW) {
    if ((tid & 31) == 0) {
      MmaState st;
      for (int q = 0; q < nets.count && ok; ++q)
        ok = mma_tiles<H>(bars, tc::smem_u32(sm), tc::smem_u32(sm + S::OFF_B), tmem, nets.n[q].image,
                          my_tiles(tiles, q), st);
      if (!ok) {
        tc::mma_commit(&bars->acc);  // drain what is in flight; nobody waits on it any more
        tc::mbar_wait(&bars->acc, st.ph_acc, tc::kDrainNs);
        atomicExch(d.err, 1u);
        atomicExch(d.err + 1, 710u);
      }
    }
    __syncwarp();
  } else {
    uint32_t ph = 0, ph_af = 0;
    for (int q = 0; q < nets.count && ok; ++q) {
      Net net = nets.n[q];
      const int mine = my_tiles(tiles, q), out = q == 0 ? OUT : 1;
      if (mine == 0) continue;
      float xn[XV];
      load_x<true>(d, rw, first_tile(tiles, q), in, xn);
      csync();  // the last network's weights and observations are read
      if (ws) {
        for (int i = tid; i < (in + 1) * H; i += kCT) ws[i] = __ldg(net.W1 + i);
        for (int i = tid; i < H; i += kCT) ws[(in + 1) * H + i] = __ldg(net.b2 + i);
        for (int i = tid; i < out * H; i += kCT) ws[(in + 2) * H + i] = __ldg(net.W3 + i);
        net.W1 = ws;
        net.b1 = ws + in * H;
        net.b2 = ws + (in + 1) * H;
        net.W3 = ws + (in + 2) * H;
      }
      store_x(xn, xp, xs);
      csync();
      for (int t = 0; t < mine && ok; ++t) {
        const int tile = first_tile(tiles, q) + t * (int)gridDim.x;
        const int next = t + 1 < mine ? tile + (int)gridDim.x : -1;
        ok = q == 0 ? fwd_tile<H, OUT, XV>(net, bars, sm, xs, in, xp, tile, tmem, ph, ph_af, d, rw, next)
                    : fwd_tile<H, 1, XV>(net, bars, sm, xs, in, xp, tile, tmem, ph, ph_af, d, rw, next);
        ph ^= 1u;
      }
    }
  }
  tc::fence_before_sync();
  __syncthreads();
  if (warp == kCW) {
    tc::fence_after_sync();
    tc::tmem_dealloc(tmem, H);
  }
}

int sm_count() {
  int dev = 0, sms = 148;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return sms;
}

template <int H, int OUT, int XV>
cudaError_t run_fwd_x(const Dev &d, const Rows &rw, int in, const Nets &nets, cudaStream_t st) {
  if (in > XV * kXT) return cudaErrorInvalidValue;
  const int xp = (in + 3) & ~3, out = OUT > 1 ? OUT : 1, smem = FwdSmem<H>::bytes(in, xp, out);
  const int off_w = FwdSmem<H>::w_fits(in, xp, out) ? FwdSmem<H>::off_w(xp) : 0;
  // (one limit for every input width: another thread's launch may come between these two)
  cudaError_t e = set_smem_limit(k_train_fwd<H, OUT, XV>, kSmemPerCta);
  if (e != cudaSuccess) return e;
  const int tiles = nets.count * (int)((rw.rows + kRows - 1) / kRows), ctas = 2 * sm_count();
  return launch_kernel(k_train_fwd<H, OUT, XV>, dim3(tiles < ctas ? tiles : ctas), dim3(kThreads), smem, st, d,
                       rw, in, xp, off_w, nets);
}
template <int H, int OUT>
cudaError_t run_fwd(const Dev &d, const Rows &rw, int in, const Nets &nets, cudaStream_t st) {
  if (in <= 2 * kXT) return run_fwd_x<H, OUT, 2>(d, rw, in, nets, st);
  if (in <= 8 * kXT) return run_fwd_x<H, OUT, 8>(d, rw, in, nets, st);
  return run_fwd_x<H, OUT, 12>(d, rw, in, nets, st);
}

// The input widths that occur with each output width of the envs' policies: 2 outputs
// with 1 or 4 inputs (landscape, control), 3 with 6 (acrobot), 10 and 20 with 5, 10 or 16
// (landscape, economy); any with the critic and with the output layer left out.
template <int H>
cudaError_t run_fwd_h(const Dev &d, const Rows &rw, int in, int out, const Nets &nets, cudaStream_t st) {
  switch (out) {
    case 1: return run_fwd<H, 1>(d, rw, in, nets, st);
    case 2: return run_fwd_x<H, 2, 2>(d, rw, in, nets, st);
    case 3: return run_fwd_x<H, 3, 8>(d, rw, in, nets, st);
    case 10: return run_fwd_x<H, 10, 8>(d, rw, in, nets, st);
    case 20: return run_fwd_x<H, 20, 8>(d, rw, in, nets, st);
    default: return run_fwd<H, 0>(d, rw, in, nets, st);
  }
}

template <int H>
void pack(const TrainGroup &g, uint8_t *img, bool back, cudaStream_t st) {
  const size_t o = g.pol.layer_offset(1), b = Geo<H>::IMAGE;
  const dim3 grid((H * H + 1023) / 1024, 2);
  k_pack_w2<H><<<grid, 256, 0, st>>>(g.params + o, g.critic + o, img, b, 0);
  if (back) k_pack_w2<H><<<grid, 256, 0, st>>>(g.params + o, g.critic + o, img + 2 * b, b, 1);
}

}  // namespace

// The fused kernels take equal hidden widths of 64, 128 or 256 units and up to 24
// inputs (the tile's observations beside the operand tiles in shared memory).
bool train_tc_supported(const PolicyShape &p) {
  return p.w[1] == p.w[2] && (p.w[1] == 64 || p.w[1] == 128 || p.w[1] == 256) && p.w[0] <= 24;
}
// Output widths of the policies that k_train_fwd holds; others run the output
// layer as a kernel of its own after it.
bool train_fwd_has_out(int out) { return out == 1 || out == 2 || out == 3 || out == 10 || out == 20; }

size_t train_image_bytes(const PolicyShape &p) {
  return train_tc_supported(p) ? (size_t)4 * 4 * p.w[1] * p.w[1] : 0;
}

void launch_train_pack(const TrainGroup &g, uint8_t *img, bool back, cudaStream_t st) {
  if (g.pol.w[1] == 64) pack<64>(g, img, back, st);
  else if (g.pol.w[1] == 128) pack<128>(g, img, back, st);
  else pack<256>(g, img, back, st);
}

// Both networks of a group, or the critic alone.
cudaError_t launch_train_fwd(const Dev &d, const TrainGroup &g, const TrainBufs &tb, uint64_t q0,
                             uint32_t n, uint32_t rows, int critic_only, cudaStream_t st) {
  const PolicyShape &p = g.pol;
  const int H = p.w[1];
  auto net = [&](const float *par, const PolicyShape &s, const uint8_t *img, float *h1, float *h2, float *out) {
    const float *W1 = par, *W2 = par + s.layer_offset(1), *W3 = par + s.layer_offset(2);
    return Net{W1, W1 + s.w[0] * H, W2 + H * H, W3, W3 + (size_t)H * s.w[3], img, h1, h2, out};
  };
  const size_t ib = (size_t)4 * H * H;
  const Net actor = net(g.params, g.pol, tb.image, tb.h1, tb.h2, tb.out);
  const Net critic = net(g.critic, g.crit, tb.image + ib, tb.c1, tb.c2, tb.vout);
  Nets nets;
  nets.n[0] = critic_only ? critic : actor;
  nets.n[1] = critic;
  nets.count = critic_only ? 1 : 2;
  const int out = critic_only ? 1 : p.w[3];
  const Rows rw{q0, n, rows, g.slot0, g.n_slots};
  if (H == 64) return run_fwd_h<64>(d, rw, p.w[0], out, nets, st);
  if (H == 128) return run_fwd_h<128>(d, rw, p.w[0], out, nets, st);
  return run_fwd_h<256>(d, rw, p.w[0], out, nets, st);
}

}  // namespace ws
