// ws_train_tc.cuh -- shared pieces of the fused update kernels (ws_train_fwd.cu,
// ws_train_bwd.cu): row tiles, the split-BF16 operand tiles and the warp roles.
//
// A CTA owns 128-row tiles of a chunk: 8 compute warps and one warp that loads
// the packed weight image and issues the MMAs.  Compute warp w works on rows 16 w
// .. + 16; its lanes lie along the units (16 lanes x 4 units = a 64-unit K block, two
// rows at a time), so that every activation row is read and written in whole
// 128-byte lines and sums over rows stay in a thread.  A K block's operand is
// handed to the MMA warp as soon as all warps have written it, and takes the place
// of the block before once its products are done.
//
// A tile is a chain of phases, each bound by something else (loads, tanhf on the
// SFU, the products, the staging of the accumulator), so two CTAs share an SM and
// overlap: with one CTA of 16 warps a tile and network of 256 units took 35 K cycles
// forward and 38 K backward, against 15 K and 10 K issue cycles and 8 K of MMAs.
#pragma once

#include "ws_kernels.cuh"
#include "ws_tc.cuh"

namespace ws {
namespace ttc {

constexpr int kRows = 128;            // rows per tile (MMA M)
constexpr int kCW = 8;                // compute warps
constexpr int kCT = 32 * kCW;         // compute threads
constexpr int kThreads = kCT + 32;    // and the MMA warp
constexpr int kWR16 = kRows / kCW;    // rows per compute warp

// Operand and staging geometry of a hidden width H (both layers).
template <int H>
struct Geo {
  static constexpr int KB = H / 64;                    // K blocks of the A operand
  static constexpr int TILE = kRows * 128;             // one K block, 128B-swizzled rows
  static constexpr int A_BYTES = 2 * TILE;             // the block in work: hi, lo
  static constexpr int NC = H / 16;                    // K = 16 chunks of the weight image
  static constexpr int CHUNK = 2 * H * 32;             // a chunk: hi [H][16], lo [H][16]
  static constexpr int NSB = 4;                        // chunk buffers
  static constexpr int B_BYTES = NSB * CHUNK;
  static constexpr int CTW = 64;                       // accumulator columns per epilogue pass
  static constexpr int CP = CTW + 4;                   // row stride of the staged accumulator
  static constexpr int CT_BYTES = kRows * CP * 4;
  static constexpr int REG = A_BYTES > CT_BYTES ? A_BYTES : CT_BYTES;
  static constexpr int IMAGE = NC * CHUNK;             // bytes of the packed image
};
constexpr int kSmemPerCta = 115712;  // two CTAs per SM

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
__device__ __forceinline__ void csync() { asm volatile("bar.sync 1, 256;" ::: "memory"); }
__device__ __forceinline__ bool call(bool v) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.u32 p, %1, 0;\n\t"
      "bar.red.and.pred q, 1, 256, p;\n\t"
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
// Store columns c .. c + 3 (c % 4 == 0) of row r of the K block in work as hi and lo.
__device__ __forceinline__ void store_a(uint32_t a, int r, int c, const float (&v)[4]) {
  uint32_t hi[2], lo[2];
  split4(v, hi, lo);
  const uint32_t o = a + (uint32_t)(r * 128 + (((c >> 3) ^ (r & 7)) << 4) + (c & 4) * 2);
  sts64(o, hi[0], hi[1]);
  sts64(o + kRows * 128, lo[0], lo[1]);
}

// The barriers of a CTA.  a and af move once per K block, acc once per tile.
struct Bars {
  uint64_t a;         // the K block in work is complete (one arrival per compute warp)
  uint64_t af;        // its products are done: the next block may take its place
  uint64_t full[4];   // weight chunk buffer filled
  uint64_t empty[4];  // the products that read the buffer are done
  uint64_t acc;       // the tile's accumulator is complete
  uint32_t tmem, pad;
};

__device__ __forceinline__ void bars_init(Bars *b) {
  tc::mbar_init(&b->a, kCW);
  tc::mbar_init(&b->af, 1);
  for (int i = 0; i < 4; ++i) tc::mbar_init(b->full + i, 1);
  for (int i = 0; i < 4; ++i) tc::mbar_init(b->empty + i, 1);
  tc::mbar_init(&b->acc, 1);
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

// The MMA warp's elected thread over n_tiles tiles of one network: acc[row][n] =
// sum_k A[row][k] B[n][k], each K = 16 step as hi hi + hi lo + lo hi.  State that
// carries over from network to network.
struct MmaState {
  uint32_t ph_a = 0;
  uint32_t seq = 0;  // weight chunks consumed since the start
  uint32_t ph_acc = 0;
};

// Before a compute warp writes a K block: the products of the block before.  Those
// of a tile's last block are covered by its accumulator.
__device__ __forceinline__ bool wait_block(Bars *b, int kb, uint32_t &ph_af) {
  if (kb == 0) return true;
  const bool ok = tc::mbar_wait(&b->af, ph_af, tc::kDrainNs);
  ph_af ^= 1u;
  return ok;
}

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
  uint32_t loaded = 0, done = 0;  // chunks of this network: requested, multiplied
  auto load_next = [&]() {
    const uint32_t s = (st.seq + loaded) % NSB;
    bulk_load(b_smem + s * G::CHUNK, image + (size_t)(loaded % G::NC) * G::CHUNK, G::CHUNK, b->full + s);
    ++loaded;
  };
  bool ok = true;
  while (loaded < NSB) load_next();  // total >= NC >= NSB
  for (int t = 0; t < n_tiles && ok; ++t) {
#pragma unroll 1
    for (int kb = 0; kb < G::KB && ok; ++kb) {
      ok = tc::mbar_wait(&b->a, st.ph_a, kLim);
      st.ph_a ^= 1u;
      if (!ok) break;
      tc::fence_after_sync();
#pragma unroll 1
      for (int q = 0; q < 4; ++q) {
        const uint32_t g = st.seq + done, s = g % NSB;
        if (!tc::mbar_wait(b->full + s, (g / NSB) & 1u, kLim)) {
          ok = false;
          break;
        }
        const uint32_t ao = a_smem + (uint32_t)(q * 32), bo = b_smem + s * G::CHUNK;
        const uint64_t ahi = tc::smem_desc(ao, 16, 1024, tc::kSwizzle128B);
        const uint64_t alo = tc::smem_desc(ao + G::TILE, 16, 1024, tc::kSwizzle128B);
        const uint64_t bhi = tc::smem_desc(bo, 128, 256, tc::kSwizzleNone);
        const uint64_t blo = tc::smem_desc(bo + H * 32, 128, 256, tc::kSwizzleNone);
        tc::mma_bf16(tmem, ahi, bhi, idesc, kb > 0 || q > 0);
        tc::mma_bf16(tmem, ahi, blo, idesc, true);
        tc::mma_bf16(tmem, alo, bhi, idesc, true);
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
      if (ok && kb + 1 < G::KB) tc::mma_commit(&b->af);
    }
    if (ok) tc::mma_commit(&b->acc);
  }
  // no copy may still be running when the CTA leaves
  for (uint32_t c = done; c < loaded; ++c) {
    const uint32_t g = st.seq + c;
    tc::mbar_wait(b->full + g % NSB, (g / NSB) & 1u, kLim);
  }
  st.seq += total;
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
  uint64_t t, s;
  if (q >> 32) {
    t = q / rw.ns;
    s = q % rw.ns;
  } else {  // 32-bit division
    t = (uint32_t)q / rw.ns;
    s = (uint32_t)q % rw.ns;
  }
  *row = (size_t)((d.k[0] - rw.n + t) % d.ring_steps);
  return rw.slot0 + (size_t)s;
}

// The tile's observations for xs[row][xp], rows past the end zero, or with REPEAT the last
// row's (a zero input times an infinite weight is NaN, which would reach the sums over the
// tile's rows through that row's zero gradients; the last row's activations are as finite
// as the sums): thread (row = tid % 128, tid / 128) takes inputs tid / 128, + 2, ...;
// loaded into registers while the tile before is still in work, then stored.
constexpr int kXT = kCT / kRows;  // threads per row
// (XV inputs per thread: as many as the network has over kXT)
template <bool REPEAT, int XV>
__device__ __forceinline__ void load_x(const Dev &d, const Rows &rw, int tile, int in, float (&v)[XV]) {
  const int tid = threadIdx.x, r = tid & 127;
  uint32_t i = (uint32_t)tile * kRows + (uint32_t)r;
  if (REPEAT) i = min(i, rw.rows - 1u);
  size_t row = 0, s = 0;
  const bool ok = i < rw.rows;
  if (ok) s = ring_slot(d, rw, i, &row);
#pragma unroll
  for (int u = 0; u < XV; ++u) {
    const int k = (tid >> 7) + kXT * u;
    v[u] = (ok && k < in) ? __ldg(d.r_obs + (row * in + k) * d.n_slots + s) : 0.f;
  }
}
template <int XV>
__device__ __forceinline__ void store_x(const float (&v)[XV], int xp, float *xs) {
  const int tid = threadIdx.x, r = tid & 127;
#pragma unroll
  for (int u = 0; u < XV; ++u) {
    const int k = (tid >> 7) + kXT * u;
    if (k < xp) xs[r * xp + k] = v[u];
  }
}

}  // namespace ttc
}  // namespace ws
