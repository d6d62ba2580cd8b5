// ws_force.cu -- the landscape force F = -grad E(x') of recorded transitions
// (FP32 SIMT path).
//
// Paper grounding: App. C builds the catalytic-reaction environment on a
// first-principles potential energy landscape of the atomic positions; the
// force on the atoms is the negative gradient of that energy.  For the
// Gaussian-sum stand-in E(x) = sum_m a_m exp(-|x - c_m|^2 / (2 w_m^2)),
//   F(x) = -grad E(x) = sum_m a_m e_m (x - c_m) / w_m^2,  e_m = exp(-|x - c_m|^2 / (2 w_m^2)).
// ws_forces evaluates it at the post-step state x' = x + dx of the last n
// steps, both recorded in the ring (obs and action), and writes the FORCE
// field [t][D][slot].  It is a scan over the ring like the returns: the roll-out
// kernels are unchanged and pay nothing when forces are not asked for.
//
// This file holds the FP32 kernel (plain and batched-FP32 paths, and the BF16
// path where the tensor-core kernel of ws_land_tc.cu does not apply, i.e.
// without the fused roll-out kernel's energy image): four threads per (step,
// env) row, a quarter of the Gaussians each, the direct difference form in registers,
// Gaussians staged through shared memory 128 at a time; each quarter tile's partial
// sums are added to the thread's running sum once per tile, and the four threads'
// sums in order (grouping keeps the FP32 error near 32 + M/128 roundings rather
// than M).
#include "ws_kernels.cuh"

namespace ws {

namespace {

constexpr int kFRows = 64;   // rows (step, env) per block
constexpr int kFG = 4;       // thread groups per block, a quarter of every tile's Gaussians each
constexpr int kFT = kFRows * kFG;
constexpr int kFTileM = 128; // Gaussians staged per tile
constexpr int kFPart = kFTileM / kFG;

// DM >= D coordinates in registers, the centres staged with zeros past D (a zero
// difference adds nothing), so that a Gaussian's coordinates are DM / 4 broadcast
// loads of 16 bytes and nothing is predicated.  Bound by the FP32 pipe: 3 D operations
// and ~12 more per pair; 32,768 rows, D 24, 4,096 Gaussians: 526 us (floor 290 us);
// with scalar, predicated loads, one thread per row and exposed tile loads 894 us.
// (Registers are held to two blocks per SM up to D 24: 128, with 64 bytes spilled.  D over
// 32 spills 476 at 255 registers: 4,096 rows, D 40 and 64, 1,000 Gaussians: 207 and 211 us,
// one thread per row 490 and 501.)
template <int DM>
__global__ __launch_bounds__(kFT, DM <= 24 ? 2 : 1) void k_force_f32(Dev d, uint32_t n) {
  __shared__ __align__(16) float cs[kFTileM * DM];      // centres (then the groups' sums)
  static_assert(kFTileM >= kFRows, "a group's sums fit");
  __shared__ float ps[kFTileM], qs[kFTileM];            // a_m / w_m^2, 1 / (2 w_m^2)
  // Gaussians whose distance and exponential chains overlap, as far as registers go
  constexpr int kFM = DM <= 32 ? 2 : 1;
  const int D = (int)d.dim;
  const size_t N = d.n_envs, S = d.n_slots;
  const int lr = threadIdx.x % kFRows, g = threadIdx.x / kFRows;
  const size_t q = (size_t)blockIdx.x * kFRows + lr;
  const bool valid = q < (size_t)n * N;
  const uint32_t i = valid ? (uint32_t)(q / N) : 0u;
  const uint32_t e = valid ? (uint32_t)(q % N) : 0u;
  const uint64_t k = d.k[0] - n + i;  // step of this row
  const size_t rowR = (size_t)(k % d.ring_steps);
  const float *obs = d.r_obs + rowR * D * S + e;
  const float *act = (const float *)d.r_act + rowR * D * S + e;
  uint64_t y[DM / 2], F[DM / 2];  // coordinate pairs
#pragma unroll
  for (int j = 0; j < DM; j += 2) {
    float x[2];
#pragma unroll
    for (int u = 0; u < 2; ++u)  // x' = x + dx in FP32, as the step computed it
      x[u] = (valid && j + u < D) ? obs[(size_t)(j + u) * S] + act[(size_t)(j + u) * S] : 0.f;
    y[j / 2] = f2_pack(x[0], x[1]);
    F[j / 2] = 0ull;
  }
  const int M = (int)d.n_gauss;
  // the next tile in registers while this one is in work: elements t, t + kFT, ... of
  // [m][DM] (zeros past D and past the last Gaussian, whose amplitude is 0 there)
  constexpr int NV = kFTileM * DM / kFT;
  float nv[NV], np = 0.f, nq = 0.f;
  auto fetch = [&](int m0) {
    const int nt = min(kFTileM, M - m0);
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      const int idx = threadIdx.x + v * kFT, m = idx / DM, j = idx % DM;
      nv[v] = m < nt && j < D ? -__ldg(d.centres + (size_t)(m0 + m) * D + j) : 0.f;  // y + (-c)
    }
    if (threadIdx.x < kFTileM) {
      const bool in = (int)threadIdx.x < nt;
      const float w = in ? __ldg(d.widths + m0 + threadIdx.x) : 1.f;
      const float iw2 = 1.0f / (w * w);
      np = in ? __ldg(d.amps + m0 + threadIdx.x) * iw2 : 0.f;
      nq = 0.5f * iw2;
    }
  };
  fetch(0);
  for (int m0 = 0; m0 < M; m0 += kFTileM) {
    const int nt = min(kFTileM, M - m0);
    __syncthreads();
#pragma unroll
    for (int v = 0; v < NV; ++v) cs[threadIdx.x + v * kFT] = nv[v];
    if (threadIdx.x < kFTileM) {
      ps[threadIdx.x] = np;
      qs[threadIdx.x] = nq;
    }
    __syncthreads();
    if (m0 + kFTileM < M) fetch(m0 + kFTileM);
    uint64_t T[DM / 2];
#pragma unroll
    for (int j = 0; j < DM / 2; ++j) T[j] = 0ull;
#pragma unroll 1
    for (int m = g * kFPart; m < min(nt, (g + 1) * kFPart); m += kFM) {
      uint64_t dd[kFM][DM / 2];
      float p[kFM];
#pragma unroll
      for (int v = 0; v < kFM; ++v) {
        uint64_t d01 = 0ull, d23 = 0ull;  // four chains, summed in a fixed order
#pragma unroll
        for (int j = 0; j < DM / 2; j += 2) {
          const ulonglong2 c = *(const ulonglong2 *)(cs + (m + v) * DM + 2 * j);
          dd[v][j] = f2_add(y[j], c.x);
          dd[v][j + 1] = f2_add(y[j + 1], c.y);
          d01 = f2_fma(dd[v][j], dd[v][j], d01);
          d23 = f2_fma(dd[v][j + 1], dd[v][j + 1], d23);
        }
        const float2 a = f2_unpack(d01), b = f2_unpack(d23);
        p[v] = ps[m + v] * expf(-((a.x + a.y) + (b.x + b.y)) * qs[m + v]);
      }
#pragma unroll
      for (int v = 0; v < kFM; ++v) {  // Gaussians in order
        const uint64_t pp = f2_pack(p[v], p[v]);
#pragma unroll
        for (int j = 0; j < DM / 2; ++j) T[j] = f2_fma(pp, dd[v][j], T[j]);
      }
    }
#pragma unroll
    for (int j = 0; j < DM / 2; ++j) F[j] = f2_add(F[j], T[j]);
  }
  // the groups' sums of a row, in order: groups 1 to 3 hand theirs over, [j][row]
  __syncthreads();
  float *out = d.r_force + rowR * D * S + e;
#pragma unroll 1
  for (int h = 1; h < kFG; ++h) {
    uint64_t *fs = (uint64_t *)cs;
    if (g == h)
#pragma unroll
      for (int j = 0; j < DM / 2; ++j) fs[j * kFRows + lr] = F[j];
    __syncthreads();
    if (g == 0)
#pragma unroll
      for (int j = 0; j < DM / 2; ++j) F[j] = f2_add(F[j], fs[j * kFRows + lr]);
    __syncthreads();
  }
  if (!valid || g) return;
#pragma unroll
  for (int j = 0; j < DM; ++j) {
    const float2 f = f2_unpack(F[j / 2]);
    if (j < D) out[(size_t)j * S] = (j & 1) ? f.y : f.x;
  }
}

template <int DM>
cudaError_t launch_f32(const Dev &d, uint32_t n, cudaStream_t st) {
  const size_t rows = (size_t)n * d.n_envs;
  return launch_kernel(k_force_f32<DM>, dim3((unsigned)((rows + kFRows - 1) / kFRows)), dim3(kFT), 0, st, d, n);
}

}  // namespace

cudaError_t launch_forces(const Dev &d, uint32_t n_steps, cudaStream_t st) {
  if (n_steps == 0) return cudaSuccess;
  // BF16 path with the fused kernel's energy image: tensor cores
  if (d.fimg) return launch_force_tc(d, d.limg, d.fimg, n_steps, st);
  if (d.dim <= 8) return launch_f32<8>(d, n_steps, st);
  if (d.dim <= 16) return launch_f32<16>(d, n_steps, st);
  if (d.dim <= 24) return launch_f32<24>(d, n_steps, st);
  if (d.dim <= 32) return launch_f32<32>(d, n_steps, st);
  return launch_f32<64>(d, n_steps, st);
}

}  // namespace ws
