// Pieces shared by the tensor-core kernels of the forward (fs_tc_fwd.cu) and the
// backward (fs_tc_bwd.cu): tile constants, the operand images and their prep
// kernels, block bookkeeping, the logits MMA chain, the slice-weight helpers and
// the host-side tensor maps, splits and launch helpers.  Internal linkage: every
// translation unit that includes it gets its own copy.
#pragma once

#include "fs_launch.h"
#include "fs_tc.h"
#include "fs_tc_ptx.cuh"

#include <cuda_bf16.h>
#include <cudaTypedefs.h>
#include <mutex>

namespace fs {
namespace {

using namespace tc;

constexpr int kThreads = 384;     // kernels with two softmax warpgroups
constexpr int kTile = 128;        // points per tile
constexpr int kGC = 128;          // slots per logits block
constexpr int kD = 32;            // head width of the tensor-core path
constexpr int kSoftmaxWarp0 = 4;  // warps 4 and up: two to four softmax warpgroups
constexpr int kStages = 3;        // x-tile pipeline depth of the deslice
constexpr int kSliceStages = 8;   // slice pipeline depth (it streams x, F and px for every 128 slots)
constexpr int kSBuf = 3;          // S buffers (logits run up to two blocks ahead)
constexpr uint32_t kXBytes = kTile * 64;   // 128 points x 32 bf16
constexpr uint32_t kExBytes = kTile * 32;  // 128 rows x 16 bf16
constexpr uint32_t kFBlock = kTile * 32;   // 128 points x 16 channels
constexpr uint32_t kPxBytes = kTile * 16;  // 128 point-extra rows of 8 bf16 (k = 0..7)
constexpr uint64_t kWaitNs = 2000000000ull;

// ---- operand images written by the prep kernels -------------------------------------------
// W image for head h (kWRow = 160 bytes per slot): G rows (slots) x 64 B of
// W' = W*log2e/tau rounded to bf16 (64B swizzle), then G rows x 32 B of
// [b'_hi, b'_lo, 1, 1, 0...] (32B swizzle), then G rows x 64 B of the residual
// W' - bf16(W') rounded to bf16 (64B swizzle).  The statistics and slice passes
// use both halves of W' (their lse, tokens and weight sums then carry no
// systematic per-slot rounding of the weights); the deslice uses the first half.
constexpr uint32_t kWRow = 160;
__device__ __forceinline__ uint32_t off_sw64(int row, int k) {  // k in [0, 32)
  const int chunk = k >> 3;
  return (uint32_t)((row >> 3) * 512 + (row & 7) * 64 + ((chunk ^ ((row & 7) >> 1)) << 4) + (k & 7) * 2);
}
__device__ __forceinline__ uint32_t off_sw32(int row, int k) {  // k in [0, 16)
  const int chunk = k >> 3;
  return (uint32_t)((row >> 3) * 256 + (row & 7) * 32 + ((chunk ^ ((row & 7) >> 2)) << 4) + (k & 7) * 2);
}
// Z' image for (b,h): blocks of 64 slots, each 32 rows (channels) x 128 B (128B swizzle).
__device__ __forceinline__ uint32_t off_z(int c, int g) {
  const int kb = g >> 6, w = g & 63;
  return (uint32_t)(kb * 4096 + (c >> 3) * 1024 + (c & 7) * 128 + (((w >> 3) ^ (c & 7)) << 4) + (w & 7) * 2);
}

// One launch prepares everything a call's passes read: its blocks are divided among jobs
// (images of W and of the tokens, point rows, splits of fp32 points, a buffer to clear), in
// the order below.  Each job alone is a few microseconds of launch and latency, and a small
// call used to spend more time in them than in its passes (a training step at N = 32,768,
// G = 64: 29 small kernels of 165 us beside 180 us of passes).
//
// Images cover slots [0, Gp), Gp = G rounded up to whole 128-slot blocks.  Padding slots
// [G, Gp) have W' = 0 and b' = -1e30 (their logits are -1e30 and their weights exactly 0 in
// every pass) and zero token rows.
constexpr int kSplitPieces = 4, kRowsPerBlock = 1024;
struct Prep {
  // blocks of 256 threads up to and including each job
  int64_t e_w, e_wt, e_t, e_z, e_px, e_split0, e_split1, e_zero;
  const float *W, *bias, *tau, *t /* tokens [BH][G][32] */, *lse, *split_src[2];
  uint8_t *wimg, *wtimg, *timg, *zimg;
  uint4* px;
  __nv_bfloat16 *split_hi[2], *split_lo[2];
  float4* zero;
  int64_t BH, N, Np, n_split8, n_zero4;
  int H, G, Gp, z_lo /* zimg with the residual half */, reset;
  uint32_t* status;
};

__device__ __forceinline__ bool good_tau(float t) { return t > 0.f && t < INFINITY; }
__device__ __forceinline__ float masked_bias(float b) { return b < kMaskedBias ? kMaskedBias : b; }
// 8 floats -> 8 bf16 (hi) and the bf16 of the residuals (lo).
__device__ __forceinline__ void split8(const float (&v)[8], uint4& hi, uint4& lo) {
  uint32_t h[4], l[4];
#pragma unroll
  for (int e = 0; e < 4; e++) {
    h[e] = pack_bf16(v[2 * e], v[2 * e + 1]);
    l[e] = pack_bf16(v[2 * e] - __uint_as_float(h[e] << 16), v[2 * e + 1] - __uint_as_float(h[e] & 0xFFFF0000u));
  }
  hi = make_uint4(h[0], h[1], h[2], h[3]);
  lo = make_uint4(l[0], l[1], l[2], l[3]);
}
__device__ __forceinline__ void load8(const float* p, float (&v)[8]) {
  const float4 a = reinterpret_cast<const float4*>(p)[0], b = reinterpret_cast<const float4*>(p)[1];
  v[0] = a.x, v[1] = a.y, v[2] = a.z, v[3] = a.w, v[4] = b.x, v[5] = b.y, v[6] = b.z, v[7] = b.w;
}

// W image, thread (h, q, g): for q < 4 the 16-byte pieces of channels [8q, 8q + 8) of slot g
// in both halves of W'; for q = 4 the slot's extra row [b'_hi, b'_lo, 1, 1, 1, 0 ...]
// (k = 2, 3, 4 multiply the three bf16 parts of the point side's -lse2, zero in the
// statistics pass).  Consecutive threads take consecutive slots, so the reads of W
// [H, d, G] coalesce.
__device__ __forceinline__ void prep_w_piece(const Prep& a, int64_t i) {
  if (i >= (int64_t)a.H * 5 * a.Gp) return;
  const int g = (int)(i % a.Gp), q = (int)((i / a.Gp) % 5), h = (int)(i / ((int64_t)5 * a.Gp));
  if (!good_tau(a.tau[h])) return;
  const float scale = kLog2e / a.tau[h];
  const bool real = g < a.G;
  uint8_t* base = a.wimg + (size_t)h * a.Gp * kWRow;
  if (q < 4) {
    float v[8];
#pragma unroll
    for (int e = 0; e < 8; e++) v[e] = real ? a.W[((int64_t)h * kD + 8 * q + e) * a.G + g] * scale : 0.f;
    const uint32_t off = off_sw64(g, 8 * q);
    split8(v, *reinterpret_cast<uint4*>(base + off), *reinterpret_cast<uint4*>(base + (size_t)a.Gp * 96 + off));
    return;
  }
  const float b2 = real ? masked_bias(a.bias[(int64_t)h * a.G + g] * scale) : -1e30f;
  const uint32_t bp = pack_bf16(b2, 0.f) & 0xFFFFu;
  const float bhi = __uint_as_float(bp << 16);
  const uint32_t blo = pack_bf16(b2 - bhi, 0.f) & 0xFFFFu;
  uint8_t* ep = base + (size_t)a.Gp * 64;
  *reinterpret_cast<uint4*>(ep + off_sw32(g, 0)) = make_uint4(bp | (blo << 16), 0x3F803F80u, 0x3F80u, 0u);
  *reinterpret_cast<uint4*>(ep + off_sw32(g, 8)) = make_uint4(0u, 0u, 0u, 0u);
}
// W'^T image of head h in the Z layout (channel rows, slots along K): the bf16 half, then
// the residual half (Gp*128 bytes per head).  Thread (h, c, 8 slots).
__device__ __forceinline__ void prep_wt_piece(const Prep& a, int64_t i) {
  const int n8 = a.Gp / 8;
  if (i >= (int64_t)a.H * kD * n8) return;
  const int g = (int)(i % n8) * 8, c = (int)((i / n8) % kD), h = (int)(i / ((int64_t)kD * n8));
  if (!good_tau(a.tau[h])) return;
  const float scale = kLog2e / a.tau[h];
  float v[8];
#pragma unroll
  for (int e = 0; e < 8; e++) v[e] = g + e < a.G ? a.W[((int64_t)h * kD + c) * a.G + g + e] * scale : 0.f;
  uint8_t* base = a.wtimg + (size_t)h * a.Gp * 128 + off_z(c, g);
  split8(v, *reinterpret_cast<uint4*>(base), *reinterpret_cast<uint4*>(base + (size_t)a.Gp * 64));
}
// T image of tokens without an added column (c = 0), in the W image's layout.
__device__ __forceinline__ void prep_t_piece(const Prep& a, int64_t i) {
  if (i >= a.BH * 5 * a.Gp) return;
  const int g = (int)(i % a.Gp), q = (int)((i / a.Gp) % 5);
  const int64_t bh = i / ((int64_t)5 * a.Gp);
  uint8_t* base = a.timg + (size_t)bh * a.Gp * kWRow;
  if (q < 4) {
    float v[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    if (g < a.G) load8(a.t + (bh * a.G + g) * kD + 8 * q, v);
    const uint32_t off = off_sw64(g, 8 * q);
    split8(v, *reinterpret_cast<uint4*>(base + off), *reinterpret_cast<uint4*>(base + (size_t)a.Gp * 96 + off));
    return;
  }
  uint8_t* ep = base + (size_t)a.Gp * 64;
  *reinterpret_cast<uint4*>(ep + off_sw32(g, 0)) = make_uint4(0u, 0x3F803F80u, 0x3F80u, 0u);
  *reinterpret_cast<uint4*>(ep + off_sw32(g, 8)) = make_uint4(0u, 0u, 0u, 0u);
}
// Z-layout image of tokens (blocks of 64 slots, 32 channel rows x 128 B, 128B swizzle): the
// bf16 half, with z_lo then the residual half.  Thread (bh, 8 slots, channel).
__device__ __forceinline__ void prep_z_piece(const Prep& a, int64_t i) {
  const int n8 = a.Gp / 8;
  if (i >= a.BH * n8 * kD) return;
  const int c = (int)(i % kD), g = (int)((i / kD) % n8) * 8;
  const int64_t bh = i / ((int64_t)kD * n8);
  float v[8];
#pragma unroll
  for (int e = 0; e < 8; e++) v[e] = g + e < a.G ? a.t[(bh * a.G + g + e) * kD + c] : 0.f;
  uint4 hi, lo;
  split8(v, hi, lo);
  uint8_t* base = a.zimg + (size_t)bh * a.Gp * (a.z_lo ? 128 : 64) + off_z(c, g);
  *reinterpret_cast<uint4*>(base) = hi;
  if (a.z_lo) *reinterpret_cast<uint4*>(base + (size_t)a.Gp * 64) = lo;
}

__device__ __forceinline__ uint4 extra_row3(float nv);  // below

__global__ void __launch_bounds__(256) k_prep(const __grid_constant__ Prep a) {
  const int64_t zero = grid_begin();
  const int64_t blk = blockIdx.x + zero;
  if (blk == 0) {
    // The status word: cleared by the first launch of a call; bad temperatures flagged.
    int bad = 0;
    for (int h = threadIdx.x + (int)zero; h < a.H; h += 256) bad |= !good_tau(a.tau[h]);
    bad = __syncthreads_or(bad);
    if (threadIdx.x == 0) {
      if (a.reset)
        *a.status = bad ? (uint32_t)FS_ERR_BAD_TAU : 0u;
      else if (bad)
        atomicCAS(a.status, 0u, (uint32_t)FS_ERR_BAD_TAU);
    }
  }
  if (blk < a.e_w) return prep_w_piece(a, blk * 256 + threadIdx.x);
  if (blk < a.e_wt) return prep_wt_piece(a, (blk - a.e_w) * 256 + threadIdx.x);
  if (blk < a.e_t) return prep_t_piece(a, (blk - a.e_wt) * 256 + threadIdx.x);
  if (blk < a.e_z) return prep_z_piece(a, (blk - a.e_t) * 256 + threadIdx.x);
  if (blk < a.e_px) {
    // Point-extra rows [1, 1, -lse2 in three parts, 0, 0, 0]; padded points get -1e30 so that
    // their weights vanish.
    const int64_t per = (a.Np + kRowsPerBlock - 1) / kRowsPerBlock, i = blk - a.e_z, bh = i / per;
    const int64_t n0 = (i - bh * per) * kRowsPerBlock + threadIdx.x;
    float v[kRowsPerBlock / 256];
#pragma unroll
    for (int e = 0; e < kRowsPerBlock / 256; e++)
      v[e] = n0 + e * 256 < a.N ? -a.lse[bh * a.N + n0 + e * 256] * kLog2e : -1e30f;
#pragma unroll
    for (int e = 0; e < kRowsPerBlock / 256; e++)
      if (n0 + e * 256 < a.Np) a.px[bh * a.Np + n0 + e * 256] = extra_row3(v[e]);
    return;
  }
  if (blk < a.e_split1) {
    // fp32 points -> bf16 hi and residual tensors of the same layout (v = hi + lo to ~2^-16
    // relative), kSplitPieces pieces of 8 values per thread in 16-byte loads and stores.
    const int k = blk < a.e_split0 ? 0 : 1;
    const int64_t i0 = (blk - (k ? a.e_split0 : a.e_px)) * (256 * kSplitPieces) + threadIdx.x;
    float v[kSplitPieces][8];
#pragma unroll
    for (int e = 0; e < kSplitPieces; e++)
      if (i0 + e * 256 < a.n_split8) load8(a.split_src[k] + 8 * (i0 + e * 256), v[e]);
#pragma unroll
    for (int e = 0; e < kSplitPieces; e++) {
      const int64_t i = i0 + e * 256;
      if (i >= a.n_split8) break;
      uint4 hi, lo;
      split8(v[e], hi, lo);
      reinterpret_cast<uint4*>(a.split_hi[k])[i] = hi;
      reinterpret_cast<uint4*>(a.split_lo[k])[i] = lo;
    }
    return;
  }
  const int64_t i = (blk - a.e_split1) * 256 + threadIdx.x;
  if (i < a.n_zero4) a.zero[i] = make_float4(0.f, 0.f, 0.f, 0.f);
}

// ---- shared pieces -------------------------------------------------------------------------
struct Work {
  int64_t bh;      // batch * H + head
  int64_t tile0;   // first point tile of this CTA
  int ntiles;      // number of point tiles (the host keeps all point indices below 2^31)
};

// Tile i and slot block c of block q = i * nb + c, kept up to date while q walks
// with a fixed stride, so that no loop divides by the runtime block count (a
// 64-bit division per block cost as much as a block's exponentials).
struct BlockPos {
  int i, c;
  __device__ __forceinline__ BlockPos(int q0, int nb) : i(0), c(q0) {
    while (c >= nb) { c -= nb; ++i; }
  }
  __device__ __forceinline__ void step(int by, int nb) {
    c += by;
    while (c >= nb) { c -= nb; ++i; }
  }
};

// Barriers on which the warpgroup that flushes an accumulator waits for its products: tile (or
// unit) i goes into accumulator i & 1, and that one's tiles take two barriers in turn.  A parity
// wait passes at once on a barrier two phases behind.  A warpgroup at tile i has seen logits that
// were issued after the products of tile i - 4, so it knows the commits issued before those
// products, tile i - 6's; with one barrier for all tiles it would have to know tile i - 4's own,
// which stands behind the commit that let those logits go.
__host__ __device__ constexpr int acc_done_of(int i) { return 2 * (i & 1) + ((i >> 1) & 1); }
__host__ __device__ constexpr uint32_t acc_done_phase(int i) { return (uint32_t)(i >> 2) & 1u; }

// CTA (split p of unit bh) processes a contiguous range of point tiles.
__device__ __forceinline__ Work work_of(int64_t N, int splits, int p, int64_t bh) {
  Work w;
  w.bh = bh;
  const int64_t tiles = (N + kTile - 1) / kTile;
  w.tile0 = tiles * p / splits;
  w.ntiles = (int)(tiles * (p + 1) / splits - w.tile0);
  return w;
}

// The constant point-side extra block: every row [1, 1, 0 x 14] (32B swizzle).
__device__ __forceinline__ void write_const_extra(uint8_t* ex) {
  for (int r = threadIdx.x; r < kTile; r += blockDim.x) {
    const uint32_t base = smem_u32(ex) + (uint32_t)((r >> 3) * 256 + (r & 7) * 32);
    const uint32_t sw = (uint32_t)((r & 7) >> 2);
    st_shared_v4(base + ((0u ^ sw) << 4), 0x3F803F80u, 0u, 0u, 0u);
    st_shared_v4(base + ((1u ^ sw) << 4), 0u, 0u, 0u, 0u);
  }
}

// Low descriptor words of the two kinds of point-side extra block: the constant one
// (32B swizzle, kHi32) and the per-tile one loaded by TMA (no swizzle, kHiPx; the k = 0..7
// core matrices at px, the zero k = 8..15 half kPxBytes further on).
__device__ __forceinline__ uint32_t const_extra_lo(uint32_t ex_s) { return sdesc_lo(ex_s, 16); }
__device__ __forceinline__ uint32_t point_extra_lo(uint32_t px_s) { return sdesc_lo(px_s, kPxBytes); }
__device__ __forceinline__ void zero_smem(uint8_t* p, uint32_t bytes) {
  for (uint32_t o = threadIdx.x * 16; o < bytes; o += blockDim.x * 16) st_shared_v4(smem_u32(p) + o, 0u, 0u, 0u, 0u);
}

// Base-2 logits of 128 points x 128 slots into TMEM.  Operands by their low descriptor
// words:
//   kPointMajor: A = points (x tile), B = slots (W);  else A = slots, B = points.
//   x, xe: the point tile and its extra block (kXeHi: its high word); w, we: the slot block's
//   W' rows and extra rows; wl: the residual half of W' (0: bf16 W' only, K = 48; else K = 80);
//   xr: the residual half of x, fp32 inputs (0: none; else two more K-steps, x_r W'_hi).
template <bool kPointMajor, uint32_t kXeHi>
__device__ __forceinline__ void issue_logits(uint32_t tmem_d, uint32_t x, uint32_t xe, uint32_t w, uint32_t we,
                                             uint32_t wl, uint32_t xr) {
  constexpr uint32_t idesc = idesc_bf16(128, kGC, false, false);
  auto mma = [&](uint32_t pt, uint32_t sl, uint32_t acc) {
    mma_ss_w<kHi64, kHi64>(tmem_d, kPointMajor ? pt : sl, kPointMajor ? sl : pt, idesc, acc);
  };
  mma(x, w, 0);
  mma(x + 2, w + 2, 1);
  if (wl) {
    mma(x, wl, 1);
    mma(x + 2, wl + 2, 1);
  }
  if (xr) {
    mma(xr, w, 1);
    mma(xr + 2, w + 2, 1);
  }
  if (kPointMajor)
    mma_ss_w<kXeHi, kHi32>(tmem_d, xe, we, idesc, 1);
  else
    mma_ss_w<kHi32, kXeHi>(tmem_d, we, xe, idesc, 1);
}

// Producer-side bulk loads of an image into smem (pieces of at most 32 KB).
__device__ __forceinline__ void load_images(uint8_t* dst, const uint8_t* src, uint32_t bytes, uint64_t* bar) {
  constexpr uint32_t kPiece = 32768;
  for (uint32_t off = 0; off < bytes; off += kPiece) {
    const uint32_t n = (bytes - off) < kPiece ? (bytes - off) : kPiece;
    bulk_load(dst + off, src + off, n, bar);
  }
}

// Slots [g0, g0 + n) of a slot image (W or T layout, Gi slots in all): the bf16 rows, the
// extra rows and, with `lo`, the residual rows, one after the other.
__device__ __forceinline__ void load_slots(uint8_t* dst, const uint8_t* img, int Gi, int g0, int n, bool lo,
                                           uint64_t* bar) {
  load_images(dst, img + (size_t)g0 * 64, (uint32_t)n * 64, bar);
  load_images(dst + (size_t)n * 64, img + (size_t)Gi * 64 + (size_t)g0 * 32, (uint32_t)n * 32, bar);
  if (lo) load_images(dst + (size_t)n * 96, img + (size_t)Gi * 96 + (size_t)g0 * 64, (uint32_t)n * 64, bar);
}

// 2^t for 32 log2-weights -> 16 bf16x2 words.
__device__ __forceinline__ void weights32(const uint32_t (&v)[32], uint32_t (&p)[16]) {
#pragma unroll
  for (int k = 0; k < 16; k++) p[k] = pack_bf16(ex2(__uint_as_float(v[2 * k])), ex2(__uint_as_float(v[2 * k + 1])));
}

// The bf16 halves hi and lo = bf16(w - hi) of a pair of weights.
__device__ __forceinline__ void split_pair(uint64_t w2, uint32_t& hi, uint32_t& lo) {
  const uint64_t neg1 = pack2(__float_as_uint(-1.f), __float_as_uint(-1.f));
  hi = pack_bf16(lo_f(w2), hi_f(w2));
  const uint64_t r2 = fma2(pack2(hi << 16, hi & 0xFFFF0000u), neg1, w2);
  lo = pack_bf16(lo_f(r2), hi_f(r2));
}

// 2^t for 32 log2-weights -> the bf16 pairs (hi) and the bf16 pairs of the
// residuals w - hi (lo): w = hi + lo to ~2^-16 relative.
__device__ __forceinline__ void weights32_hilo(const uint32_t (&v)[32], uint32_t (&hi)[16], uint32_t (&lo)[16]) {
#pragma unroll
  for (int k = 0; k < 16; k++) {
    const uint64_t w2 = pack2(__float_as_uint(ex2(__uint_as_float(v[2 * k]))),
                              __float_as_uint(ex2(__uint_as_float(v[2 * k + 1]))));
    split_pair(w2, hi[k], lo[k]);
  }
}

// 64 log2-weights of one TMEM lane in columns [0, 64) from tS -> bf16 weights packed in
// pairs into columns [0, 32) from tP (which may be columns this thread has read).
__device__ __forceinline__ void weights_half(uint32_t tS, uint32_t tP) {
  uint32_t v0[32], v1[32];
  tmem_ld32(tS, v0);
  tmem_ld32(tS + 32, v1);
  tmem_wait_ld2(v0, v1);
  uint32_t pk0[16], pk1[16];
  weights32(v0, pk0);
  weights32(v1, pk1);
  tmem_st16(tP, pk0);
  tmem_st16(tP + 16, pk1);
}

// Split products: 32 columns of log2-weights -> in place the bf16 weights packed in pairs
// (16 columns), then the bf16 pairs of their residuals (16).
__device__ __forceinline__ void weights32_hilo_inplace(uint32_t tS) {
  uint32_t v[32], hi[16], lo[16];
  tmem_ld32(tS, v);
  tmem_wait_ld(v);
  weights32_hilo(v, hi, lo);
  tmem_st16(tS, hi);
  tmem_st16(tS + 16, lo);
}
// TMEM column, within a run of such packed columns, of the hi pairs of K-step kk (16
// entries); their lo pairs are 16 columns on.
__device__ __forceinline__ uint32_t da_col(int kk) { return (uint32_t)(32 * (kk >> 1) + 8 * (kk & 1)); }
// One 64-column half.  (With 64 columns in registers at a time the fp32 deslice call at
// N = 262,144, H = 8, G = 512 took 402 us against 372.)
__device__ __forceinline__ void weights_hilo_half(uint32_t tS) {
  weights32_hilo_inplace(tS);
  weights32_hilo_inplace(tS + 32);
}

// The same, plus acc += sum over the half's 64 slots of w_g ds[g] (ds: the half's slice of a
// per-slot array in shared memory; every lane reads the same address, a broadcast).  The
// backward of the slice needs this sum for its delta (the dS term).  The loop stays rolled:
// unrolled, the sums of one 32 overlap the next and spill at 128 registers a thread (whole
// backward at B = 2, N = 131,072, H = 8, G = 512 1926 us against 1850).
__device__ __forceinline__ void weights32_hilo_ds(const uint32_t (&v)[32], uint32_t (&hi)[16], uint32_t (&lo)[16],
                                                  const float* ds, float& acc) {
  const float4* d4 = reinterpret_cast<const float4*>(ds);
#pragma unroll
  for (int k = 0; k < 8; k++) {
    const float4 q = d4[k];
    float w[4];
#pragma unroll
    for (int e = 0; e < 4; e++) w[e] = ex2(__uint_as_float(v[4 * k + e]));
    acc = fmaf(w[0], q.x, acc);
    acc = fmaf(w[1], q.y, acc);
    acc = fmaf(w[2], q.z, acc);
    acc = fmaf(w[3], q.w, acc);
#pragma unroll
    for (int e = 0; e < 2; e++)
      split_pair(pack2(__float_as_uint(w[2 * e]), __float_as_uint(w[2 * e + 1])), hi[2 * k + e], lo[2 * k + e]);
  }
}
__device__ __forceinline__ void weights_hilo_half_ds(uint32_t tS, const float* ds, float& acc) {
#pragma unroll 1
  for (int e = 0; e < 64; e += 32) {
    uint32_t v[32], hi[16], lo[16];
    tmem_ld32(tS + e, v);
    tmem_wait_ld(v);
    weights32_hilo_ds(v, hi, lo, ds + e, acc);
    tmem_st16(tS + e, hi);
    tmem_st16(tS + e + 16, lo);
  }
}

// A point-extra row [1, 1, -v_1, -v_2, -v_3, 0, 0, 0] (bf16): v = v_1 + v_2 + v_3 in
// three bf16 parts, which hold v's 24 significant bits, so that the row adds -v to
// fp32 precision against a slot side [.., .., 1, 1, 1, 0 ...].  (Two parts would
// leave an error of ~2^-17 |v|: as -lse2, a per-point error of the weights'
// normalisation, which the softmax backward's cancellation amplifies in dtau.)
__device__ __forceinline__ uint4 extra_row3(float nv) {
  const __nv_bfloat16 p1 = __float2bfloat16_rn(nv);
  const float r1 = nv - __bfloat162float(p1);
  const __nv_bfloat16 p2 = __float2bfloat16_rn(r1);
  const __nv_bfloat16 p3 = __float2bfloat16_rn(r1 - __bfloat162float(p2));
  return make_uint4(0x3F803F80u, (uint32_t)__bfloat16_as_ushort(p1) | ((uint32_t)__bfloat16_as_ushort(p2) << 16),
                    (uint32_t)__bfloat16_as_ushort(p3), 0u);
}

// ---- host side -------------------------------------------------------------------------------
PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  });
  return fn;
}

// 3-D view of a [B, N, C] bf16 tensor; box = (box_c channels, 128 points, 1).
bool make_point_map(CUtensorMap* map, const void* ptr, const Shape& s, int box_c, CUtensorMapSwizzle sw) {
  auto fn = encode_fn();
  if (!fn) return false;
  const uint64_t C = (uint64_t)s.H * s.d;
  cuuint64_t dims[3] = {C, (cuuint64_t)s.N, (cuuint64_t)s.B};
  cuuint64_t strides[2] = {C * 2, (cuuint64_t)s.N * C * 2};
  cuuint32_t box[3] = {(cuuint32_t)box_c, (cuuint32_t)kTile, 1};
  cuuint32_t estr[3] = {1, 1, 1};
  return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(ptr), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, sw, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// 2-D view of the point-extra rows [B*H*Np, 8] bf16; box = (8, 128 points).
bool make_px_map(CUtensorMap* map, const void* ptr, int64_t BH, int64_t Np) {
  auto fn = encode_fn();
  if (!fn) return false;
  cuuint64_t dims[2] = {8, (cuuint64_t)(BH * Np)};
  cuuint64_t strides[1] = {16};
  cuuint32_t box[2] = {8, (cuuint32_t)kTile};
  cuuint32_t estr[2] = {1, 1};
  return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(ptr), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// The tensor-core kernels see G rounded up to whole 128-slot blocks (padding slots
// carry weight 0); outputs keep the caller's G.
Shape tc_padded(const Shape& s) {
  Shape r = s;
  r.G = (s.G + kGC - 1) / kGC * kGC;
  return r;
}

size_t w_image_bytes(const Shape& s) { return (size_t)s.H * s.G * kWRow; }
// Z' image of the forward's deslice; fp32 inputs carry z' as hi and residual halves.
size_t z_image_bytes(const Shape& s) { return (size_t)s.BH() * s.G * (s.dtype == FS_F32 ? 128 : 64); }
int64_t padded_n(const Shape& s) { return (s.N + kTile - 1) / kTile * kTile; }
size_t px_bytes(const Shape& s) { return (size_t)s.BH() * padded_n(s) * 16; }

// Point splits P per work unit for one-CTA-per-SM kernels: the P that minimises the makespan
// waves * (tiles a split * blocks + kFixedBlocks), where a tile is `blocks` blocks of 0.35 to
// 0.6 us and a CTA's start and end (set-up, images, first loads, last products, partial rows)
// cost as much as kFixedBlocks.  Measured: statistics and deslice 2.6 and 2.9 us, slice 4.7 to
// 6.  Counting whole waves alone takes P = 19 for most shapes, up to eight waves of short CTAs
// (against P = 6 at B = 3, N = 20,011, G = 100: statistics 24.4 us against 19.2, slice 33.3
// against 23.8, deslice 27.1 against 21.3, backward 235 against 184; slice against P = 7 at
// B = 1, N = 262,144, G = 1024 374 against 355; the other way round statistics at B = 4,
// N = 262,144, G = 256: 351 at P = 19, 362 at 9).  P is no larger than whole waves alone would
// take it, and at most one split per point tile, which bounds the partials' workspace.
constexpr int kFixedBlocks = 8;
// The P of the fewest whole waves per split alone, smallest on ties.
int wave_splits(const Shape& s, int units) {
  const int64_t tiles = (s.N + kTile - 1) / kTile, sms = num_sms();
  int64_t best = 1;
  double best_t = 1e30;
  for (int64_t p = 1; p <= 2 * sms && p <= tiles; p++) {
    const double t = (double)((units * p + sms - 1) / sms) / (double)p;
    if (t < best_t - 1e-12) {
      best_t = t;
      best = p;
    }
  }
  return (int)best;
}
int point_splits(const Shape& s, int units, int blocks) {
  const int64_t tiles = (s.N + kTile - 1) / kTile, sms = num_sms();
  if (units < 1) units = 1;
  const int64_t most = wave_splits(s, units);
  int64_t best = 1, best_t = INT64_MAX;
  for (int64_t p = 1; p <= most; p++) {
    const int64_t t = (units * p + sms - 1) / sms * ((tiles + p - 1) / p * blocks + kFixedBlocks);
    if (t < best_t) {
      best_t = t;
      best = p;
    }
  }
  return (int)best;
}

constexpr size_t kMaxSmem = 232448;  // opt-in shared memory per block on sm_103
template <typename K>
cudaError_t set_smem(K kernel, size_t bytes) {
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

// A call's preparation: jobs are added in any order, run() launches them as one kernel.
struct Prepare {
  Prep a{};
  int64_t w = 0, wt = 0, t = 0, z = 0, px = 0, sp[2] = {0, 0}, zero = 0;  // threads of each job
  // sp.G: slots of the images, G: the caller's.
  Prepare(const Shape& sp_, int G, const float* tau, uint32_t* status, bool reset) {
    a.H = sp_.H, a.G = G, a.Gp = sp_.G, a.BH = sp_.BH(), a.N = sp_.N, a.Np = padded_n(sp_);
    a.tau = tau, a.status = status, a.reset = reset ? 1 : 0;
  }
  void weights(const float* W, const float* bias, uint8_t* img) {
    a.W = W, a.bias = bias, a.wimg = img;
    w = (int64_t)a.H * 5 * a.Gp;
  }
  void weights_t(const float* W, uint8_t* img) {
    a.W = W, a.wtimg = img;
    wt = (int64_t)a.H * kD * (a.Gp / 8);
  }
  void tokens(const float* tok, uint8_t* timg, uint8_t* zimg, bool z_lo) {
    a.t = tok, a.timg = timg, a.zimg = zimg, a.z_lo = z_lo ? 1 : 0;
    t = timg ? a.BH * 5 * a.Gp : 0;
    z = a.BH * (a.Gp / 8) * kD;
  }
  void rows(const float* lse, void* dst) {
    a.lse = lse, a.px = static_cast<uint4*>(dst);
    px = a.BH * ((a.Np + kRowsPerBlock - 1) / kRowsPerBlock) * 256;
  }
  // fp32 points v -> bf16 hi at dst, residuals at dst + half.
  void split(const Shape& s, const void* v, uint8_t* dst, size_t half) {
    const int k = sp[0] ? 1 : 0;
    a.split_src[k] = static_cast<const float*>(v);
    a.split_hi[k] = reinterpret_cast<__nv_bfloat16*>(dst);
    a.split_lo[k] = reinterpret_cast<__nv_bfloat16*>(dst + half);
    a.n_split8 = s.B * s.N * s.H * s.d / 8;
    sp[k] = (a.n_split8 + kSplitPieces - 1) / kSplitPieces;
  }
  void clear(float* p, int64_t n) {  // n rounded up to 4 floats
    a.zero = reinterpret_cast<float4*>(p);
    a.n_zero4 = zero = (n + 3) / 4;
  }
  cudaError_t run(cudaStream_t st) {
    int64_t e = 0;
    auto end = [&](int64_t threads) { return e += (threads + 255) / 256; };
    a.e_w = end(w), a.e_wt = end(wt), a.e_t = end(t), a.e_z = end(z), a.e_px = end(px);
    a.e_split0 = end(sp[0]), a.e_split1 = end(sp[1]), a.e_zero = end(zero);
    return launch(k_prep, dim3((unsigned)(e > 0 ? e : 1)), dim3(256), 0, st, a);
  }
};

}  // namespace
}  // namespace fs
