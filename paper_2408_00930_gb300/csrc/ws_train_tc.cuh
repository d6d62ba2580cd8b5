// ws_train_tc.cuh -- shared pieces of the fused update kernels (ws_train_fwd.cu,
// ws_train_bwd.cu): row tiles, the split-BF16 operand tiles and the warp roles.
//
// A CTA owns 128-row tiles of a chunk: 16 compute warps and one warp that loads
// the packed weight image and issues the MMAs.  Compute warp w works on rows 8 w
// .. + 8; its lanes lie along the units (16 lanes x 4 units = a 64-unit K block, two
// rows at a time), so that every activation row is read and written in whole
// 128-byte lines and sums over rows stay in a thread.  A K block's operand is
// handed to the MMA warp as soon as all warps have written it, so the products run
// under the CUDA-core work of the following blocks.
#pragma once

#include "ws_kernels.cuh"
#include "ws_tc.cuh"

namespace ws {
namespace ttc {

constexpr int kRows = 128;            // rows per tile (MMA M)
constexpr int kCW = 16;               // compute warps
constexpr int kCT = 32 * kCW;         // compute threads
constexpr int kThreads = kCT + 32;    // and the MMA warp

// Operand and staging geometry of a hidden width H (both layers).
template <int H>
struct Geo {
  static constexpr int KB = H / 64;                    // K blocks of the A operand
  static constexpr int TILE = kRows * 128;             // one K block, 128B-swizzled rows
  static constexpr int A_BYTES = 2 * KB * TILE;        // hi blocks, lo blocks
  static constexpr int NC = H / 16;                    // K = 16 chunks of the weight image
  static constexpr int CHUNK = 2 * H * 32;             // a chunk: hi [H][16], lo [H][16]
  static constexpr bool RES = H <= 128;                // the whole image stays in shared memory
  static constexpr int NSB = RES ? NC : 5;             // chunk buffers (streamed: 5 x 16 KB)
  static constexpr int B_BYTES = NSB * CHUNK;
  static constexpr int CTW = H < 128 ? H : 128;        // accumulator columns per epilogue pass
  static constexpr int CP = CTW + 4;                   // row stride of the staged accumulator
  static constexpr int CT_BYTES = kRows * CP * 4;
  static constexpr int REG = A_BYTES > CT_BYTES ? A_BYTES : CT_BYTES;
  static constexpr int IMAGE = NC * CHUNK;             // bytes of the packed image
};

__device__ __forceinline__ void bulk_load(uint32_t dst, const void *src, uint32_t bytes,
                                          uint64_t *bar) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(tc::smem_u32(bar)),
               "r"(bytes)
               : "memory");
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
          dst),
      "l"(src), "r"(bytes), "r"(tc::smem_u32(bar))
      : "memory");
}
__device__ __forceinline__ void arrive(uint64_t *bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(tc::smem_u32(bar)) : "memory");
}
// Barrier (and AND vote) of the compute warps.
__device__ __forceinline__ void csync() { asm volatile("bar.sync 1, 512;" ::: "memory"); }
__device__ __forceinline__ bool call(bool v) {
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
__device__ __forceinline__ void sts64(uint32_t addr, uint32_t a, uint32_t b) {
  asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(addr), "r"(a), "r"(b) : "memory");
}
// Split four values into BF16 hi and lo words (x = hi + lo to about 2^-17 |x|).
__device__ __forceinline__ void split4(const float (&v)[4], uint32_t (&hi)[2], uint32_t (&lo)[2]) {
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    hi[j] = tc::pack_bf16x2(v[2 * j], v[2 * j + 1]);
    lo[j] = tc::pack_bf16x2(v[2 * j] - tc::bf16_lo(hi[j]), v[2 * j + 1] - tc::bf16_hi(hi[j]));
  }
}
// Store columns c .. c + 3 (c % 4 == 0) of K block kb of row r as hi and lo.
template <int H>
__device__ __forceinline__ void store_a(uint32_t a, int kb, int r, int c, const float (&v)[4]) {
  uint32_t hi[2], lo[2];
  split4(v, hi, lo);
  const uint32_t o = a + (uint32_t)(kb * Geo<H>::TILE + r * 128 + (((c >> 3) ^ (r & 7)) << 4) + (c & 4) * 2);
  sts64(o, hi[0], hi[1]);
  sts64(o + Geo<H>::KB * Geo<H>::TILE, lo[0], lo[1]);
}

// The barriers of a CTA.
struct Bars {
  uint64_t a[4];     // K block kb of the A operand is complete (one arrival per compute warp)
  uint64_t full[5];  // weight chunk buffer filled (resident weights: full[0], the image)
  uint64_t empty[5]; // streamed weights: the MMAs that read the buffer are done
  uint64_t acc;      // the tile's accumulator is complete
  uint32_t tmem, pad;
};

__device__ __forceinline__ void bars_init(Bars *b) {
  for (int i = 0; i < 4; ++i) tc::mbar_init(b->a + i, kCW);
  for (int i = 0; i < 5; ++i) tc::mbar_init(b->full + i, 1);
  for (int i = 0; i < 5; ++i) tc::mbar_init(b->empty + i, 1);
  tc::mbar_init(&b->acc, 1);
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

// The MMA warp's elected thread over n_tiles tiles of one network: acc[row][n] =
// sum_k A[row][k] B[n][k], each K = 16 step as hi hi + hi lo + lo hi.  State that
// carries over from network to network.
struct MmaState {
  uint32_t ph_a = 0;      // phase of the a[] barriers (all move once per tile)
  uint32_t ph_full = 0;   // resident weights: phase of full[] (once per network)
  uint32_t seq = 0;       // streamed weights: chunks consumed since the start
  uint32_t ph_acc = 0;
};

template <int H>
__device__ __forceinline__ bool mma_tiles(Bars *b, uint32_t a_smem, uint32_t b_smem, uint32_t tmem,
                                          const uint8_t *__restrict__ image, int n_tiles,
                                          MmaState &st) {
  using G = Geo<H>;
  constexpr uint32_t idesc = tc::idesc_bf16_f32(kRows, H);
  constexpr uint64_t kLim = tc::kDrainNs;
  constexpr uint32_t NSB = G::NSB;
  if (n_tiles <= 0) return true;
  const uint32_t total = (uint32_t)n_tiles * G::NC;
  uint32_t loaded = 0, done = 0;  // streamed chunks of this network: requested, multiplied
  auto load_next = [&]() {
    const uint32_t s = (st.seq + loaded) % NSB;
    bulk_load(b_smem + s * G::CHUNK, image + (size_t)(loaded % G::NC) * G::CHUNK, G::CHUNK, b->full + s);
    ++loaded;
  };
  bool ok = true;
  if (G::RES) {
    bulk_load(b_smem, image, G::IMAGE, b->full);
    ok = tc::mbar_wait(b->full, st.ph_full, kLim);
    st.ph_full ^= 1u;
  } else {
    while (loaded < NSB) load_next();  // total >= NC > NSB
  }
  for (int t = 0; t < n_tiles && ok; ++t) {
#pragma unroll 1
    for (int kb = 0; kb < G::KB && ok; ++kb) {
      ok = tc::mbar_wait(b->a + kb, st.ph_a, kLim);
      if (!ok) break;
      tc::fence_after_sync();
#pragma unroll 1
      for (int q = 0; q < 4; ++q) {
        const int c = 4 * kb + q;
        const uint32_t g = st.seq + done;
        const uint32_t s = G::RES ? (uint32_t)c : g % NSB;
        if (!G::RES && !tc::mbar_wait(b->full + s, (g / NSB) & 1u, kLim)) {
          ok = false;
          break;
        }
        const uint32_t ao = a_smem + (uint32_t)(kb * G::TILE + q * 32);
        const uint32_t bo = b_smem + s * G::CHUNK;
        const uint64_t ahi = tc::smem_desc(ao, 16, 1024, tc::kSwizzle128B);
        const uint64_t alo = tc::smem_desc(ao + G::KB * G::TILE, 16, 1024, tc::kSwizzle128B);
        const uint64_t bhi = tc::smem_desc(bo, 128, 256, tc::kSwizzleNone);
        const uint64_t blo = tc::smem_desc(bo + H * 32, 128, 256, tc::kSwizzleNone);
        tc::mma_bf16(tmem, ahi, bhi, idesc, c > 0);
        tc::mma_bf16(tmem, ahi, blo, idesc, true);
        tc::mma_bf16(tmem, alo, bhi, idesc, true);
        if (!G::RES) {
          tc::mma_commit(b->empty + s);
          // refill the buffer of the chunk before: its products end while this
          // chunk's are queued behind them
          if (done > 0 && loaded < total) {
            const uint32_t gp = g - 1;
            if (!tc::mbar_wait(b->empty + gp % NSB, (gp / NSB) & 1u, kLim)) {
              ok = false;
              break;
            }
            load_next();
          }
          ++done;
        }
      }
    }
    if (ok) tc::mma_commit(&b->acc);
    st.ph_a ^= 1u;
  }
  if (!G::RES) {
    // no copy may still be running when the CTA leaves
    for (uint32_t c = done; c < loaded; ++c) {
      const uint32_t g = st.seq + c;
      tc::mbar_wait(b->full + g % NSB, (g / NSB) & 1u, kLim);
    }
    st.seq += total;
  }
  // the last tile's products (and with them every buffer's) are done before the
  // next network's weights arrive
  st.ph_acc ^= (uint32_t)(n_tiles - 1) & 1u;
  if (ok) ok = tc::mbar_wait(&b->acc, st.ph_acc, kLim);
  st.ph_acc ^= 1u;
  return ok;
}

// One pass of the accumulator (columns c0 .. c0 + CTW) from tensor memory into
// ct[row][CP] by the compute warps (warp w: lanes 32 (w % 4).., 32 columns at
// 32 (w / 4)).
template <int H>
__device__ __forceinline__ void stage_acc(uint32_t tmem, float *ct, int c0, int warp, int lane) {
  using G = Geo<H>;
  const int cg = warp >> 2;
  if (cg * 32 >= G::CTW) return;
  uint32_t z[32];
  tc::tmem_ld32(tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(c0 + cg * 32), z);
  tc::tmem_wait_ld();
  float *o = ct + ((warp & 3) * 32 + lane) * G::CP + cg * 32;
#pragma unroll
  for (int i = 0; i < 32; i += 4)
    *(float4 *)(o + i) = make_float4(__uint_as_float(z[i]), __uint_as_float(z[i + 1]),
                                     __uint_as_float(z[i + 2]), __uint_as_float(z[i + 3]));
}

// Tiles of network q of a launch: the (network, tile) pairs go to the CTAs round
// robin, network by network.
__device__ __forceinline__ int first_tile(int tiles, int q) {
  const int g = (int)gridDim.x, o = ((int)blockIdx.x - q * tiles) % g;
  return o < 0 ? o + g : o;
}
__device__ __forceinline__ int my_tiles(int tiles, int q) {
  const int f = first_tile(tiles, q);
  return f < tiles ? (tiles - f + (int)gridDim.x - 1) / (int)gridDim.x : 0;
}

// Ring position of row i of the chunk that starts at global row q0 of a group.
struct Rows {
  uint64_t q0;
  uint32_t n, rows, slot0, ns;
};
__device__ __forceinline__ size_t ring_slot(const Dev &d, const Rows &rw, uint32_t i, size_t *row) {
  const uint64_t q = rw.q0 + i;
  const uint64_t k = d.k[0] - rw.n + q / rw.ns;
  *row = (size_t)(k % d.ring_steps);
  return rw.slot0 + (size_t)(q % rw.ns);
}

// The tile's observations into xs[row][XP] (rows past the end: zeros).
__device__ __forceinline__ void gather_x(const Dev &d, const Rows &rw, int tile, int in, int xp,
                                         float *xs) {
  const int tid = threadIdx.x, r = tid & 127;
  const uint32_t i = (uint32_t)tile * kRows + (uint32_t)r;
  size_t row = 0, s = 0;
  const bool ok = i < rw.rows;
  if (ok) s = ring_slot(d, rw, i, &row);
  for (int k = tid >> 7; k < xp; k += kCT / 128)
    xs[r * xp + k] = (ok && k < in) ? d.r_obs[(row * in + k) * d.n_slots + s] : 0.f;
}

}  // namespace ttc
}  // namespace ws
