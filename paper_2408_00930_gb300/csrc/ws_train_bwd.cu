// ws_train_bwd.cu -- fused backward pass of the actor-critic update: the data
// gradients and the narrow layers' weight gradients in one launch, the
// hidden-by-hidden weight gradient in a second, all slice sums in a third.
//
// Paper grounding: Sec. 2 and App. B keep the training step on the GPU beside the
// roll-out store.
//
// k_train_bwd, per 128-row tile: d2 = (dout W3^T) (1 - h2^2) in FP32 FMAs (outputs
// in order from zero), written for the weight gradient and split into BF16 hi + lo
// operand tiles; dW3 = h2^T dout while the products run; d1 = (d2 W2^T) (1 - h1^2)
// from the accumulator and dW1 = x^T d1 at once, so that d1 never leaves the SM.
// Sums over rows run thread by thread (a column and a group of rows each), then
// over groups, tiles and CTAs in fixed orders.  k_train_wgrad: dW2 = h1^T d2 over
// row slices with both operands split into row-major ("MN-major") tiles straight
// from the row-major activations, and db2 as the loader's column sums.  The parts
// ran as ten kernels per network that passed each activation through memory seven
// times.  A chunk of 58,368 rows of 4-256-256-2, both networks: k_train_bwd 109 us
// (bound by the tails of its phases, DRAM 42% busy), k_train_wgrad 61 us (by its loads;
// 35 us at the copy bandwidth), k_train_reduce 21 us; layer by layer 106 and 66 us per
// network for the two wide products alone.
#include "ws_train_tc.cuh"

namespace ws {

namespace {

using namespace ttc;

// Rows on their way into L2 ahead of their loads (16-byte aligned, a multiple of 16 bytes).
__device__ __forceinline__ void prefetch_l2(const float *p, uint32_t bytes) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}

struct BNet {
  const float *W3, *h1, *h2, *dout;
  float *d2;
  const uint8_t *image;  // packed W2, backward operand
  float *p1, *p3;        // this network's CTA partials [cta][(in + 1) H], [cta][(H + 1) out]
};
struct BNets {
  BNet n[2];
  int count;
};

// XP: inputs rounded up to 4; OUT: outputs (0: d2 is given, dW3 is formed elsewhere).
template <int H, int XP, int OUT>
struct BwdSmem {
  using G = Geo<H>;
  static constexpr int SL1 = kCT * (XP + 1) * 4;       // dW1's group sums, over the operand tile
  static constexpr int REG = G::REG > SL1 ? G::REG : SL1;
  static constexpr int OFF_B = (REG + 1023) / 1024 * 1024;
  static constexpr int OFF_BAR = OFF_B + G::B_BYTES;
  static constexpr int OFF_X = OFF_BAR + ((int)sizeof(Bars) + 15) / 16 * 16;  // [128][XP]
  static constexpr int OFF_D = OFF_X + kRows * XP * 4;                          // [128][OUT]
  static constexpr int OFF_W3 = OFF_D + (kRows * OUT * 4 + 15) / 16 * 16;       // [OUT][H]
  static constexpr int OFF_A3 = OFF_W3 + OUT * H * 4;                           // [(H + 1) OUT]
  static constexpr int OFF_A1 = OFF_A3 + ((H + 1) * OUT * 4 + 15) / 16 * 16;    // [(XP + 1) H]
  static constexpr int WITH_A1 = OFF_A1 + (XP + 1) * H * 4 + 1024;
  static constexpr bool A1_SMEM = WITH_A1 <= kSmemPerCta;  // else the dW1 sums stay in global memory
  static constexpr int BYTES = A1_SMEM ? WITH_A1 : OFF_A1 + 1024;
  static_assert(BYTES <= kSmemPerCta, "shared memory of half an SM");
};

// One tile of one network by the compute warps; a1, a3 the CTA's running sums.
template <int H, int XP, int OUT, bool A1S>
__device__ __forceinline__ bool bwd_tile(const BNet &net, Bars *bars, uint8_t *reg, const float *xs,
                                         float *ds, const float *w3t, float *a1, float *a3, int in,
                                         int rows, int tile, uint32_t tmem, uint32_t ph_acc,
                                         uint32_t &ph_af) {
  using G = Geo<H>;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int l16 = lane & 15, rh = lane >> 4;
  const uint32_t a = tc::smem_u32(reg);
  const size_t row0 = (size_t)tile * kRows;
  // ---- d2, one 64-unit K block at a time
  bool okw = true;
  const float *src = (OUT > 0 ? net.h2 : net.d2) + (row0 + warp * kWR16 + rh) * H + l16 * 4;
  float4 hn[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) hn[i] = __ldg((const float4 *)(src + 2 * i * H));
#pragma unroll 1
  for (int it = 0; it < 2 * G::KB; ++it) {  // half a block (eight rows per warp) at a time
    const int kb = it >> 1, i0 = (it & 1) * 8, col = kb * 64 + l16 * 4;
    float4 h[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) h[i] = hn[i];
    if (it + 1 < 2 * G::KB) {  // the next half's loads run under this half's work
      const float *nx = src + ((it + 1) & 1) * 8 * H + ((it + 1) >> 1) * 64;
#pragma unroll
      for (int i = 0; i < 4; ++i) hn[i] = __ldg((const float4 *)(nx + 2 * i * H));
    }
    float s[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) s[i][j] = 0.f;
    if (OUT > 0) {
#pragma unroll(OUT > 0 && OUT <= 4 ? OUT : 4)
      for (int o = 0; o < OUT; ++o) {
        const float4 w = *(const float4 *)(w3t + o * H + col);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float dv = ds[(warp * kWR16 + i0 + 2 * i + rh) * OUT + o];
          s[i][0] = fmaf(dv, w.x, s[i][0]);
          s[i][1] = fmaf(dv, w.y, s[i][1]);
          s[i][2] = fmaf(dv, w.z, s[i][2]);
          s[i][3] = fmaf(dv, w.w, s[i][3]);
        }
      }
    }
    if (i0 == 0) okw = wait_block(bars, kb, ph_af) && okw;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int r = warp * kWR16 + i0 + 2 * i + rh;
      if (OUT > 0) {
        s[i][0] *= 1.f - h[i].x * h[i].x;
        s[i][1] *= 1.f - h[i].y * h[i].y;
        s[i][2] *= 1.f - h[i].z * h[i].z;
        s[i][3] *= 1.f - h[i].w * h[i].w;
        *(float4 *)(net.d2 + (row0 + r) * H + col) = make_float4(s[i][0], s[i][1], s[i][2], s[i][3]);
      } else {
        const bool ok = (int)row0 + r < rows;  // a partial tile's rows past the end
        s[i][0] = ok ? h[i].x : 0.f;
        s[i][1] = ok ? h[i].y : 0.f;
        s[i][2] = ok ? h[i].z : 0.f;
        s[i][3] = ok ? h[i].w : 0.f;
      }
      store_a(a, r, l16 * 4, s[i]);
    }
    if (i0) {
      tc::fence_async_smem();
      tc::fence_before_sync();
      __syncwarp();
      if (lane == 0) arrive(&bars->a);
    }
  }
  // ---- dW3 and db3 of the tile while the products run: a thread per column and share
  // of the outputs
  if (OUT > 0) {
    constexpr int TPC = kCT / H > 0 ? kCT / H : 1, O = (OUT + TPC - 1) / TPC > 0 ? (OUT + TPC - 1) / TPC : 1;
    const int c = tid % H, o0 = tid / H * O;
    if (o0 < OUT) {
      float acc[O];
#pragma unroll
      for (int o = 0; o < O; ++o) acc[o] = 0.f;
      const float *hp = net.h2 + row0 * H + c;
      constexpr int U = 16;  // loads in flight
#pragma unroll 1
      for (int r = 0; r < kRows; r += U) {
        float hv[U];
#pragma unroll
        for (int u = 0; u < U; ++u) hv[u] = __ldg(hp + (size_t)(r + u) * H);
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const float *dp = ds + (r + u) * OUT + o0;
#pragma unroll
          for (int o = 0; o < O; ++o)
            if (OUT % O == 0 || o0 + o < OUT) acc[o] = fmaf(hv[u], dp[o], acc[o]);
        }
      }
#pragma unroll
      for (int o = 0; o < O; ++o)
        if (OUT % O == 0 || o0 + o < OUT) a3[c * OUT + o0 + o] += acc[o];
    }
    for (int o = warp; o < OUT; o += kCW) {  // db3: a warp per output
      float t = 0.f;
#pragma unroll
      for (int r = 0; r < kRows; r += 32) t += ds[(r + lane) * OUT + o];
#pragma unroll
      for (int m = 16; m > 0; m >>= 1) t += __shfl_xor_sync(0xffffffffu, t, m);
      if (lane == 0) a3[H * OUT + o] += t;
    }
  }
  // ---- d1 and dW1
  const bool ok = call(tc::mbar_wait(&bars->acc, ph_acc, tc::kDrainNs) && okw);
  if (!ok) return false;
  tc::fence_after_sync();
  float *ct = (float *)reg;
#pragma unroll 1
  for (int c0 = 0; c0 < H; c0 += G::CTW) {
    constexpr int LPR = G::CTW / 4, RPW = 32 / LPR, NI = kWR16 / RPW;  // lanes per row, rows per access
    const int c = (lane % LPR) * 4;
    float4 h[NI];  // the activations' loads in flight while the accumulator is staged
#pragma unroll
    for (int i = 0; i < NI; ++i)
      h[i] = __ldg((const float4 *)(net.h1 + (row0 + warp * kWR16 + i * RPW + lane / LPR) * H + c0 + c));
    stage_acc<H>(tmem, ct, c0, warp, lane);
    tc::fence_before_sync();
    csync();
#pragma unroll
    for (int i = 0; i < NI; ++i) {
      float4 *p = (float4 *)(ct + (warp * kWR16 + i * RPW + lane / LPR) * G::CP + c);
      float4 v = *p;
      v.x *= 1.f - h[i].x * h[i].x;
      v.y *= 1.f - h[i].y * h[i].y;
      v.z *= 1.f - h[i].z * h[i].z;
      v.w *= 1.f - h[i].w * h[i].w;
      *p = v;
    }
    csync();
    constexpr int NG = kCT / G::CTW, L = kRows / NG;
    const int cc = tid % G::CTW, g = tid / G::CTW;
    float acc[XP + 1];
#pragma unroll
    for (int k = 0; k <= XP; ++k) acc[k] = 0.f;
#pragma unroll 4
    for (int r = g * L; r < g * L + L; ++r) {
      const float dv = ct[r * G::CP + cc];
#pragma unroll
      for (int k = 0; k < XP; k += 4) {
        const float4 x = *(const float4 *)(xs + r * XP + k);
        acc[k] = fmaf(x.x, dv, acc[k]);
        acc[k + 1] = fmaf(x.y, dv, acc[k + 1]);
        acc[k + 2] = fmaf(x.z, dv, acc[k + 2]);
        acc[k + 3] = fmaf(x.w, dv, acc[k + 3]);
      }
      acc[XP] += dv;
    }
    csync();
    float *sl = ct;  // [NG][XP + 1][CTW]
#pragma unroll
    for (int k = 0; k <= XP; ++k) sl[(g * (XP + 1) + k) * G::CTW + cc] = acc[k];
    csync();
    for (int v = tid; v < (in + 1) * G::CTW; v += kCT) {
      const int k = v / G::CTW, q = v % G::CTW;
      const int kk = k == in ? XP : k;  // the bias row follows the true inputs
      float t = 0.f;
#pragma unroll
      for (int u = 0; u < NG; ++u) t += sl[(u * (XP + 1) + kk) * G::CTW + q];
      if (A1S)
        a1[k * H + c0 + q] += t;
      else
        atomicAdd(a1 + k * H + c0 + q, t);  // (this thread's alone: no wait for the old value)
    }
    csync();
  }
  return true;
}

template <int H, int XP, int OUT>
__global__ void __launch_bounds__(kThreads, 2)
    k_train_bwd(Dev d, Rows rw, int in, const __grid_constant__ BNets nets) {
  using G = Geo<H>;
  using S = BwdSmem<H, XP, OUT>;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = tc::smem_u32(smem_raw);
  uint8_t *sm = smem_raw + ((1024u - (raw & 1023u)) & 1023u);
  Bars *bars = (Bars *)(sm + S::OFF_BAR);
  float *xs = (float *)(sm + S::OFF_X), *ds = (float *)(sm + S::OFF_D);
  float *w3t = (float *)(sm + S::OFF_W3), *a3 = (float *)(sm + S::OFF_A3);
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
        tc::mma_commit(&bars->acc);
        tc::mbar_wait(&bars->acc, st.ph_acc, tc::kDrainNs);
        atomicExch(d.err, 1u);
        atomicExch(d.err + 1, 711u);
      }
    }
    __syncwarp();
  } else {
    uint32_t ph = 0, ph_af = 0;
    constexpr int XV = (XP + kXT - 1) / kXT;
    for (int q = 0; q < nets.count && ok; ++q) {
      const BNet &net = nets.n[q];
      const int no = q == 0 ? OUT : (OUT > 0 ? 1 : 0);  // 0: no output layer here
      float *p1 = net.p1 + (size_t)blockIdx.x * (in + 1) * H;
      float *a1 = S::A1_SMEM ? (float *)(sm + S::OFF_A1) : p1;
      csync();
      for (int i = tid; i < (in + 1) * H; i += kCT) a1[i] = 0.f;
      for (int i = tid; i < (H + 1) * no; i += kCT) a3[i] = 0.f;
      for (int i = tid; i < no * H; i += kCT) w3t[i] = __ldg(net.W3 + (i % H) * no + i / H);
      const int mine = my_tiles(tiles, q), t0 = first_tile(tiles, q);
      float xn[XV];
      if (mine > 0) load_x<false>(d, rw, t0, in, xn);
      for (int t = 0; t < mine && ok; ++t) {
        const int tile = t0 + t * (int)gridDim.x;
        store_x(xn, XP, xs);
        for (int i = tid; i < kRows * no; i += kCT) {
          const int r = tile * kRows + i / (no > 0 ? no : 1);
          ds[i] = r < (int)rw.rows ? net.dout[(size_t)tile * kRows * no + i] : 0.f;
        }
        csync();
        if (t + 1 < mine) load_x<false>(d, rw, tile + (int)gridDim.x, in, xn);
        if (q == 0)
          ok = bwd_tile<H, XP, OUT, S::A1_SMEM>(net, bars, sm, xs, ds, w3t, a1, a3, in, (int)rw.rows,
                                                tile, tmem, ph, ph_af);
        else
          ok = bwd_tile<H, XP, (OUT > 0 ? 1 : 0), S::A1_SMEM>(net, bars, sm, xs, ds, w3t, a1, a3, in,
                                                              (int)rw.rows, tile, tmem, ph, ph_af);
        ph ^= 1u;
      }
      csync();
      if (S::A1_SMEM)
        for (int i = tid; i < (in + 1) * H; i += kCT) p1[i] = a1[i];
      float *p3 = net.p3 + (size_t)blockIdx.x * (H + 1) * no;
      for (int i = tid; i < (H + 1) * no; i += kCT) p3[i] = a3[i];
    }
  }
  tc::fence_before_sync();
  __syncthreads();
  if (warp == kCW) {
    tc::fence_after_sync();
    tc::tmem_dealloc(tmem, H);
  }
}

// ------------------------------------------------------------------ dW2, db2
// D[m][n] = sum over the slice's rows of h1[row][m0 + m] d2[row][n], M = 128 (H =
// 64: rows 64.. of the operand are zero), N = H.  Per stage of 32 rows the compute
// warps (two rows each) load float4s of both arrays two stages ahead and store them
// as hi and lo tiles in the 128B-swizzled MN-major layout: 64 units of a row are one
// 128-byte line, eight rows a swizzle atom, four atoms (32 rows) a 64-unit block.
constexpr int kWW = 16, kWC = 32 * kWW, kWT = kWC + 32;  // loader warps, their threads, and the MMA warp
constexpr int kWR = 32;   // rows per stage
constexpr int kWS = 4;    // stages
constexpr int kWPre = 2;  // stages prefetched into L2 past the two in registers
template <int H>
struct WGeo {
  static constexpr int MC = H < 128 ? H : 128;          // columns of h1 per CTA
  static constexpr int MH = H / MC;                     // CTAs (M halves) per slice
  static constexpr int ABLK = 2, BBLK = H / 64;         // 64-unit blocks of each operand
  static constexpr int BLK = kWR * 128;                 // bytes of a block
  static constexpr int A_B = ABLK * BLK, B_B = BBLK * BLK;
  static constexpr int STAGE = 2 * (A_B + B_B);         // A hi, A lo, B hi, B lo
  static constexpr int CT = kRows * 132 * 4;            // output staging over the stages
  static constexpr int REG = kWS * STAGE > CT ? kWS * STAGE : CT;
  static constexpr int OFF_CS = REG;                    // [16][H] column sums
  static constexpr int OFF_BAR = OFF_CS + kWW * H * 4;
  static constexpr int SMEM = OFF_BAR + 128 + 1024;
  static_assert(SMEM <= 232448, "shared memory over the 227 KB per-CTA limit");
};
struct WNet {
  const float *h1, *d2;
  float *part;  // [slice][(H + 1) H]
};

// idesc of kind::f16, BF16 operands both MN-major (transpose bits 15 and 16).
__device__ constexpr uint32_t idesc_mn(uint32_t N) {
  return tc::idesc_bf16_f32(128, N) | (1u << 15) | (1u << 16);
}

__device__ __forceinline__ void store_mn(uint32_t base, int r, int c, const float4 &q, uint32_t lo_off,
                                         int blk) {
  const float v[4] = {q.x, q.y, q.z, q.w};
  uint32_t hi[2], lo[2];
  split4(v, hi, lo);
  const int cc = c & 63;
  const uint32_t o = base + (uint32_t)((c >> 6) * blk + (r >> 3) * 1024 + (r & 7) * 128 +
                                       (((cc >> 3) ^ (r & 7)) << 4) + (cc & 4) * 2);
  sts64(o, hi[0], hi[1]);
  sts64(o + lo_off, lo[0], lo[1]);
}

// Barrier (and AND vote) of the loader warps.
__device__ __forceinline__ void wsync() { asm volatile("bar.sync 1, 512;" ::: "memory"); }
__device__ __forceinline__ bool wall(bool v) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.u32 p, %1, 0;\n\t"
      "bar.red.and.pred q, 1, 512, p;\n\t"
      "selp.u32 %0, 1, 0, q;\n\t}"
      : "=r"(r)
      : "r"((uint32_t)v)
      : "memory");
  return r != 0;
}

template <int H>
__global__ void __launch_bounds__(kWT, 1)
    k_train_wgrad(const __grid_constant__ WNet n0, const __grid_constant__ WNet n1, int rows, int per,
                  uint32_t *err) {
  using G = WGeo<H>;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = tc::smem_u32(smem_raw);
  uint8_t *sm = smem_raw + ((1024u - (raw & 1023u)) & 1023u);
  const uint32_t sb = tc::smem_u32(sm);
  uint64_t *full = (uint64_t *)(sm + G::OFF_BAR), *empty = full + kWS, *done = empty + kWS;
  uint32_t *holder = (uint32_t *)(done + 1);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const WNet &net = blockIdx.z ? n1 : n0;
  const int m0 = (int)blockIdx.y * G::MC, slice = (int)blockIdx.x;
  const int rb = slice * per, re = min(rows, rb + per);
  const int ns = re > rb ? (re - rb + kWR - 1) / kWR : 0;
  if (tid == 0) {
    for (int i = 0; i < kWS; ++i) {
      tc::mbar_init(full + i, kWW);
      tc::mbar_init(empty + i, 1);
    }
    tc::mbar_init(done, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (H < 128)  // the operand's unused half
    for (int i = tid; i < kWS * G::STAGE / 16; i += kWT) ((uint4 *)sm)[i] = make_uint4(0, 0, 0, 0);
  if (warp == kWW) tc::tmem_alloc(holder, H);
  tc::fence_async_smem();
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = *holder;
  bool ok = true;
  if (warp == kWW) {
    if (lane == 0 && ns > 0) {
      // This CTA's share of stage s's rows into L2: with two column halves one CTA takes
      // d2, the other h1.  The two stages in registers do not cover the loads' latency
      // while all SMs read (3.3 TB/s at 256 units); a copy into L2 needs no registers.
      // 58,368 rows, 256 units: 73.5 us without, 63.3 / 60.9 / 62.4 / 68.4 / 80.2 us
      // with 1 / 2 / 3 / 6 / 12 stages (48 us if every load hit L2).
      auto prefetch = [&](int s) {
        if (s >= ns) return;
        const int r0 = rb + s * kWR;
        const uint32_t bytes = (uint32_t)(min(kWR, re - r0) * H * 4);
        if (gridDim.y == 1 || blockIdx.y == 0) prefetch_l2(net.d2 + (size_t)r0 * H, bytes);
        if (gridDim.y == 1 || blockIdx.y == 1) prefetch_l2(net.h1 + (size_t)r0 * H, bytes);
      };
      for (int s = 2; s < 2 + kWPre; ++s) prefetch(s);
      for (int s = 0; s < ns && ok; ++s) {
        prefetch(s + 2 + kWPre);
        const int b = s % kWS;
        ok = tc::mbar_wait(full + b, (uint32_t)(s / kWS) & 1u, tc::kDrainNs);
        if (!ok) break;
        tc::fence_after_sync();
        const uint32_t st = sb + (uint32_t)(b * G::STAGE);
#pragma unroll
        for (int q = 0; q < kWR / 16; ++q) {
          const uint32_t o = (uint32_t)(q * 2048);  // two 8-row atoms per K = 16
          const uint64_t ahi = tc::smem_desc(st + o, G::BLK, 1024, tc::kSwizzle128B);
          const uint64_t alo = tc::smem_desc(st + G::A_B + o, G::BLK, 1024, tc::kSwizzle128B);
          const uint64_t bhi = tc::smem_desc(st + 2 * G::A_B + o, G::BLK, 1024, tc::kSwizzle128B);
          const uint64_t blo = tc::smem_desc(st + 2 * G::A_B + G::B_B + o, G::BLK, 1024, tc::kSwizzle128B);
          tc::mma_bf16(tmem, ahi, bhi, idesc_mn(H), s > 0 || q > 0);
          tc::mma_bf16(tmem, ahi, blo, idesc_mn(H), true);
          tc::mma_bf16(tmem, alo, bhi, idesc_mn(H), true);
        }
        tc::mma_commit(empty + b);
      }
      tc::mma_commit(done);
      if (!tc::mbar_wait(done, 0, tc::kDrainNs)) ok = false;
      if (!ok) {
        atomicExch(err, 1u);
        atomicExch(err + 1, 712u);
      }
    }
    __syncwarp();
  } else {
    // warp w: rows 2 w, 2 w + 1 of a stage; a lane's columns: 128 j + 4 lane (H >=
    // 128), or 4 (lane % 16) of row 2 w + lane / 16 (H = 64)
    constexpr int NB = H >= 128 ? 2 * (H / 128) : 1, NA = H >= 128 ? 2 : 1;
    float4 va[2][NA], vb[2][NB];  // the next two stages, in flight
    float cs[H >= 128 ? H / 128 : 1][4];
#pragma unroll
    for (int j = 0; j < (H >= 128 ? H / 128 : 1); ++j)
#pragma unroll
      for (int q = 0; q < 4; ++q) cs[j][q] = 0.f;
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
    auto load = [&](int s, float4 (&va)[NA], float4 (&vb)[NB]) {
      const int r0 = rb + s * kWR + warp * 2;
      if (H >= 128) {
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const bool in = r0 + i < re;
          va[i] = in ? __ldg((const float4 *)(net.h1 + (size_t)(r0 + i) * H + m0 + 4 * lane)) : zero;
#pragma unroll
          for (int j = 0; j < H / 128; ++j)
            vb[i * (H / 128) + j] =
                in ? __ldg((const float4 *)(net.d2 + (size_t)(r0 + i) * H + 128 * j + 4 * lane)) : zero;
        }
      } else {
        const int r = r0 + (lane >> 4);
        va[0] = r < re ? __ldg((const float4 *)(net.h1 + (size_t)r * H + 4 * (lane & 15))) : zero;
        vb[0] = r < re ? __ldg((const float4 *)(net.d2 + (size_t)r * H + 4 * (lane & 15))) : zero;
      }
    };
    auto put = [&](int s, const float4 (&va)[NA], const float4 (&vb)[NB]) {
      const uint32_t st = sb + (uint32_t)((s % kWS) * G::STAGE);
      if (H >= 128) {
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const int r = warp * 2 + i;
          store_mn(st, r, 4 * lane, va[i], G::A_B, G::BLK);
#pragma unroll
          for (int j = 0; j < H / 128; ++j) {
            const float4 q = vb[i * (H / 128) + j];
            store_mn(st + 2 * G::A_B, r, 128 * j + 4 * lane, q, G::B_B, G::BLK);
            cs[j][0] += q.x;
            cs[j][1] += q.y;
            cs[j][2] += q.z;
            cs[j][3] += q.w;
          }
        }
      } else {
        const int r = warp * 2 + (lane >> 4), c = 4 * (lane & 15);
        store_mn(st, r, c, va[0], G::A_B, G::BLK);
        store_mn(st + 2 * G::A_B, r, c, vb[0], G::B_B, G::BLK);
        cs[0][0] += vb[0].x;
        cs[0][1] += vb[0].y;
        cs[0][2] += vb[0].z;
        cs[0][3] += vb[0].w;
      }
    };
    if (ns > 0) load(0, va[0], vb[0]);
    if (ns > 1) load(1, va[1], vb[1]);
    for (int s0 = 0; s0 < ns && ok; s0 += 2) {
#pragma unroll
      for (int h = 0; h < 2; ++h) {  // the register buffers by compile-time index
        const int s = s0 + h;
        if (s >= ns || !ok) break;
        const int b = s % kWS;
        if (s >= kWS) ok = tc::mbar_wait(empty + b, (uint32_t)(s / kWS - 1) & 1u, tc::kDrainNs);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        put(s, va[h], vb[h]);
        if (s + 2 < ns) load(s + 2, va[h], vb[h]);
        tc::fence_async_smem();
        __syncwarp();
        if (lane == 0) arrive(full + b);
      }
    }
    float *csum = (float *)(sm + G::OFF_CS);
    if (H >= 128) {
#pragma unroll
      for (int j = 0; j < H / 128; ++j)
        *(float4 *)(csum + warp * H + 128 * j + 4 * lane) =
            make_float4(cs[j][0], cs[j][1], cs[j][2], cs[j][3]);
    } else {
#pragma unroll
      for (int q = 0; q < 4; ++q) cs[0][q] += __shfl_xor_sync(0xffffffffu, cs[0][q], 16);
      if (lane < 16)
        *(float4 *)(csum + warp * H + 4 * lane) = make_float4(cs[0][0], cs[0][1], cs[0][2], cs[0][3]);
    }
    float *out = net.part + (size_t)slice * ((size_t)(H + 1) * H);
    if (ns > 0) ok = tc::mbar_wait(done, 0, tc::kDrainNs) && ok;
    ok = wall(ok);
    if (ok) {
      tc::fence_after_sync();
      if (m0 == 0)
        for (int c = tid; c < H; c += kWC) {
          float t = csum[c];
#pragma unroll
          for (int w = 1; w < kWW; ++w) t += csum[w * H + c];
          out[(size_t)H * H + c] = t;
        }
      float *ct = (float *)sm;
      constexpr int CW = H < 128 ? H : 128;
#pragma unroll 1
      for (int c0 = 0; c0 < H; c0 += CW) {
        const int cg = warp >> 2;
        if (cg * 32 < CW) {
          uint32_t z[32];
          if (ns > 0) {
            tc::tmem_ld32(tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(c0 + cg * 32), z);
            tc::tmem_wait_ld();
          } else {
#pragma unroll
            for (int i = 0; i < 32; ++i) z[i] = 0u;
          }
          float *o = ct + ((warp & 3) * 32 + lane) * 132 + cg * 32;
#pragma unroll
          for (int i = 0; i < 32; i += 4)
            *(float4 *)(o + i) = make_float4(__uint_as_float(z[i]), __uint_as_float(z[i + 1]),
                                             __uint_as_float(z[i + 2]), __uint_as_float(z[i + 3]));
        }
        wsync();
        for (int i = tid; i < G::MC * CW / 4; i += kWC) {
          const int m = i / (CW / 4), c = (i % (CW / 4)) * 4;
          *(float4 *)(out + (size_t)(m0 + m) * H + c0 + c) = *(const float4 *)(ct + m * 132 + c);
        }
        wsync();
      }
    }
  }
  tc::fence_before_sync();
  __syncthreads();
  if (warp == kWW) {
    tc::fence_after_sync();
    tc::tmem_dealloc(tmem, H);
  }
}

// ------------------------------------------------------------ slice sums
// grad[i] += sum_z P[z len + i], z in a fixed order, for all layers of both networks
// in one launch: a block per 32 consecutive i (eight lanes of four where every slice
// starts on 16 bytes), 64 groups of lanes over the slices z, z + 64, ..., then the
// groups' sums in order, eight and eight.  Short chains and many blocks: the kernel
// is a latency of two loads and three barriers over the read of the partial sums.
struct Seg {
  const float *P;
  float *grad;
  int nz;
  uint32_t len, block0;
};
struct Segs {
  Seg s[6];
  int count;
};
__global__ __launch_bounds__(512) void k_train_reduce(const __grid_constant__ Segs segs) {
  __shared__ float4 part[64][8];
  __shared__ float part2[8][32];
  int q = 0;
  while (q + 1 < segs.count && blockIdx.x >= segs.s[q + 1].block0) ++q;
  const Seg &sg = segs.s[q];
  const int l = threadIdx.x & 7, g = threadIdx.x >> 3;
  const uint32_t i0 = (blockIdx.x - sg.block0) * 32, i = i0 + 4 * l;
  const bool vec = (sg.len & 3) == 0 && ((uintptr_t)sg.P & 15) == 0;
  float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 3
  for (int z = g; z < sg.nz; z += 64) {
    const float *p = sg.P + (size_t)z * sg.len + i;
    if (vec && i < sg.len) {
      const float4 v = __ldcs((const float4 *)p);
      s.x += v.x;
      s.y += v.y;
      s.z += v.z;
      s.w += v.w;
    } else if (!vec) {
      if (i < sg.len) s.x += __ldcs(p);
      if (i + 1 < sg.len) s.y += __ldcs(p + 1);
      if (i + 2 < sg.len) s.z += __ldcs(p + 2);
      if (i + 3 < sg.len) s.w += __ldcs(p + 3);
    }
  }
  part[g][l] = s;
  __syncthreads();
  const float *pf = (const float *)part;
  const int c = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (w < 8) {
    float t = pf[8 * w * 32 + c];
#pragma unroll
    for (int k = 1; k < 8; ++k) t += pf[(8 * w + k) * 32 + c];
    part2[w][c] = t;
  }
  __syncthreads();
  if (w == 0 && i0 + c < sg.len) {
    float t = sg.grad[i0 + c];
#pragma unroll
    for (int k = 0; k < 8; ++k) t += part2[k][c];
    sg.grad[i0 + c] = t;
  }
}

int sm_count() {
  int dev = 0, sms = 148;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return sms < kTrainMaxCtas / 2 ? sms : kTrainMaxCtas / 2;
}

template <int H, int XP, int OUT>
cudaError_t run_bwd(const Dev &d, const Rows &rw, int in, const BNets &nets, int grid, cudaStream_t st) {
  using S = BwdSmem<H, XP, OUT>;
  cudaError_t e = set_smem_limit(k_train_bwd<H, XP, OUT>, S::BYTES);
  if (e != cudaSuccess) return e;
  return launch_kernel(k_train_bwd<H, XP, OUT>, dim3(grid), dim3(kThreads), S::BYTES, st, d, rw, in, nets);
}

// The output widths come with their input widths (control 4 -> 2, acrobot 6 -> 3,
// economy 16 -> 20 and 10); any other pair takes d2 from a kernel before.
template <int H>
cudaError_t run_bwd_h(const Dev &d, const Rows &rw, int in, int out, const BNets &nets, int grid,
                      cudaStream_t st) {
  if (in == 4 && out == 2) return run_bwd<H, 4, 2>(d, rw, in, nets, grid, st);
  if (in == 6 && out == 3) return run_bwd<H, 8, 3>(d, rw, in, nets, grid, st);
  if constexpr (H <= 128) {
    if (in == 16 && out == 20) return run_bwd<H, 16, 20>(d, rw, in, nets, grid, st);
    if (in == 16 && out == 10) return run_bwd<H, 16, 10>(d, rw, in, nets, grid, st);
  }
  if (in <= 8) return run_bwd<H, 8, 0>(d, rw, in, nets, grid, st);
  if (in <= 16) return run_bwd<H, 16, 0>(d, rw, in, nets, grid, st);
  return run_bwd<H, 24, 0>(d, rw, in, nets, grid, st);
}

template <int H>
cudaError_t run_wgrad(const WNet &a, const WNet &c, int rows, int slices, int per, uint32_t *err,
                      cudaStream_t st) {
  using G = WGeo<H>;
  cudaError_t e = set_smem_limit(k_train_wgrad<H>, G::SMEM);
  if (e != cudaSuccess) return e;
  return launch_kernel(k_train_wgrad<H>, dim3((unsigned)slices, G::MH, 2), dim3(kWT), G::SMEM, st, a, c, rows,
                       per, err);
}

}  // namespace

bool train_bwd_has_out(const PolicyShape &p) {
  const int in = p.w[0], out = p.w[3];
  return (in == 4 && out == 2) || (in == 6 && out == 3) ||
         (p.w[1] <= 128 && in == 16 && (out == 20 || out == 10));
}

// Floats of the fused backward's partial sums (both networks).
size_t train_part_floats(const PolicyShape &p) {
  if (!train_tc_supported(p)) return 0;
  const size_t H = p.w[1];
  return 2 * ((size_t)kTrainMaxCtas * ((p.w[0] + 1) * H + (H + 1) * p.w[3]) + kTrainMaxSlices * (H + 1) * H) + 16;
}

cudaError_t launch_train_bwd(const Dev &d, const TrainGroup &g, const TrainBufs &tb, uint64_t q0,
                             uint32_t n, uint32_t rows, cudaStream_t st) {
  const PolicyShape &p = g.pol;
  const int H = p.w[1], in = p.w[0], out = p.w[3];
  const bool has = train_bwd_has_out(p);
  const int sms = sm_count(), tiles = (int)((rows + kRows - 1) / kRows);
  const int grid = tiles < sms ? 2 * tiles : 2 * sms;
  const size_t ib = (size_t)4 * H * H;
  // partials: per network p1, p3 [grid], then the dW2 slices
  const size_t l1 = (size_t)(in + 1) * H, l2 = (size_t)(H + 1) * H, l3a = (size_t)(H + 1) * out, l3c = H + 1;
  float *f = tb.part;
  auto take = [&](size_t m) { float *r = f; f += m; return r; };
  float *p1a = take(grid * l1), *p1c = take(grid * l1), *p3a = take(grid * l3a), *p3c = take(grid * l3c);
  f = tb.part + ((size_t)(f - tb.part) + 3) / 4 * 4;
  // slices of the rows: at most 1,024 rows each (what one accumulator sums), and
  // whole rounds of the SMs' CTAs where the slices are many
  const int per_round = sms / (2 * (H > 128 ? H / 128 : 1)) > 0 ? sms / (2 * (H > 128 ? H / 128 : 1)) : 1;
  int slices = ((int)rows + 1023) / 1024;
  const int up = (slices + per_round - 1) / per_round * per_round;
  if (up <= kTrainMaxSlices) slices = up;
  int per = ((int)rows + slices - 1) / slices;
  per = (per + kWR - 1) / kWR * kWR;
  slices = ((int)rows + per - 1) / per;
  float *p2a = take((size_t)slices * l2), *p2c = take((size_t)slices * l2);
  const float *W3a = g.params + g.pol.layer_offset(2), *W3c = g.critic + g.crit.layer_offset(2);
  BNets nets;
  nets.n[0] = BNet{W3a, tb.h1, tb.h2, tb.out, tb.d1, tb.image + 2 * ib, p1a, p3a};
  nets.n[1] = BNet{W3c, tb.c1, tb.c2, tb.vout, tb.d2, tb.image + 3 * ib, p1c, p3c};
  nets.count = 2;
  const Rows rw{q0, n, rows, g.slot0, g.n_slots};
  cudaError_t e = H == 64    ? run_bwd_h<64>(d, rw, in, out, nets, grid, st)
                  : H == 128 ? run_bwd_h<128>(d, rw, in, out, nets, grid, st)
                             : run_bwd_h<256>(d, rw, in, out, nets, grid, st);
  if (e != cudaSuccess) return e;
  const WNet wa{tb.h1, tb.d1, p2a}, wc{tb.c1, tb.d2, p2c};
  e = H == 64    ? run_wgrad<64>(wa, wc, (int)rows, slices, per, d.err, st)
      : H == 128 ? run_wgrad<128>(wa, wc, (int)rows, slices, per, d.err, st)
                 : run_wgrad<256>(wa, wc, (int)rows, slices, per, d.err, st);
  if (e != cudaSuccess) return e;
  Segs s;
  s.count = 0;
  uint32_t blocks = 0;
  auto seg = [&](const float *P, float *grad, int nz, size_t len) {
    s.s[s.count++] = Seg{P, grad, nz, (uint32_t)len, blocks};
    blocks += (uint32_t)((len + 31) / 32);
  };
  float *ga = tb.grad, *gc = tb.grad + g.pol.count();
  seg(p2a, ga + g.pol.layer_offset(1), slices, l2);
  seg(p2c, gc + g.crit.layer_offset(1), slices, l2);
  seg(p1a, ga, grid, l1);
  seg(p1c, gc, grid, l1);
  if (has) {
    seg(p3a, ga + g.pol.layer_offset(2), grid, l3a);
    seg(p3c, gc + g.crit.layer_offset(2), grid, l3c);
  }
  return launch_kernel(k_train_reduce, dim3(blocks), dim3(512), 0, st, s);
}

}  // namespace ws
