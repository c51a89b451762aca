// The point-by-slot passes of the SIMT path: fp32 FMA products and fp32 accumulation
// (the paper's "ieee" dot level, Appendix G.2) for d = 16, 32, 64, any G, fp32 or bf16
// point tensors.
//
// Every pass works on tiles of 128 points x TG slots as a register-tiled matrix product.
// What bounds it is the FMA pipe (128 per clock per SM; fma.f32x2 measured no more), and
// before it the shared-memory reads that feed it.  A kernel with a thread per point reads
// each slot's row as a broadcast, one 16-byte load per four FMAs; such a load takes 2.4
// clocks of an SM's shared-memory pipe and the four FMAs one, so that form stops near 40% of
// the FMA rate (it ran at 22 to 30%).  Here a thread holds 8 points x 8 slots (d = 64:
// 8 x 4) of a tile, so that 16 floats read feed 64 FMAs.  16-byte loads in which runs of
// four lanes share an address take 2.4 clocks, others 4 (measured), so in every product the
// side with more loads goes over lane >> 2 and the other over lane & 3.
//
// Measured (B = 2, N = 65,536, H = 8, d = 32, G = 256, fp32, against the thread-per-point and
// thread-per-slot kernels): statistics 0.82 -> 0.41 ms, d z' 1.50 -> 0.98, delta and dx
// 5.50 -> 2.90, dW 3.97 -> 1.69; at d = 64 (N = 16,384, H = 4, G = 64, bf16), where a point's
// rows do not fit a thread's registers, delta and dx 3.85 -> 0.15 ms.
//
// One layout serves all products of a tile, with rows padded by four floats:
//   points  [d][128 + 4]  x, dO, fx transposed (channel-major)
//   slots   [d][TG + 4]   W' (as in memory), z', dU transposed
//   weights [TG][128 + 4] w or da of the tile, between the two products of a pass
// Products (p point, g slot, c or k channel):
//   pair_products  acc[p][g] += sum_k points[k][p] slots[k][g]     logits, dw
//   point_products acc[p][c] += sum_g weights[g][p] slots[c][g]    out, dfx, dx
//   slot_products  acc[g][c] += sum_p weights[g][p] points[c][p]   U, d z', dW
//
// Ownership follows the paper's G-blocked family (Appendix G.1): point-owned passes
// (statistics, deslice, delta and dx) sweep the slot tiles; slot-owned passes (slice, dW)
// sweep the point tiles of one split and write partials, which are summed in a fixed order
// afterwards.  No float atomics.
//
// Logits are a2 = x . (W log2e/tau) + beta log2e/tau, the temperature-scaled logit in
// base-2 units, so w = exp2(a2 - lse2) with lse2 = lse log2e.  Slots past G get W = 0 and
// beta = kLowest and points past N lse2 = 1e30, and a masked slot's bias is finite (kMaskedBias):
// their weights are exactly 0 and every sum stays finite.
#pragma once

#include "fs_launch.h"
#include "fs_simt_tiles.h"

#include <cuda_bf16.h>
#include <type_traits>

namespace fs {
namespace {

constexpr int TP = kSimtTP;
constexpr int LP = TP + 4;  // row length of the point and weight tiles
constexpr float kFar = 1e30f;        // lse2 of points past N
constexpr float kLowest = -3.4e38f;  // base-2 logit of slots past G, below every masked slot's

// Threads and register tiles: with d = 64 and 64 slots one block of 256 threads fills an SM's
// shared memory, else there are two or more blocks of 128.
template <int D, int TG>
struct Tile {
  static constexpr int kThreads = D == 64 && TG == 64 ? 256 : 128;
  static constexpr int kWarps = kThreads / 32;
  static constexpr int LG = TG + 4;  // row length of the slot tiles
  // pair_products: two rows of warps over the points, 8 points per thread
  static constexpr int kPairN = TG / (4 * (kWarps / 2));
  // point_products: warps over points x channels
  static constexpr int kPtCols = D == 16 ? 1 : (D == 32 ? 2 : 4);  // warp columns of 16 channels
  static constexpr int kPtRows = kWarps / kPtCols;
  static constexpr int kPtM = TP / (8 * kPtRows);
  static constexpr int kPtN = 4;
  // slot_products: warps over two halves of the points x channels
  static constexpr int kSlM = TG / 8;
  static constexpr int kSlN = D / (2 * kWarps);
  static_assert((kPairN == 4 || kPairN == 8) && (kPtM == 4 || kPtM == 8 || kPtM == 16) && kSlN >= 1, "register tiles");

  static constexpr size_t kPointTile = (size_t)D * LP;
  static constexpr size_t kSlotTile = (size_t)D * LG;
  static constexpr size_t kWeightTile = (size_t)TG * LP;
  // write_rows goes through the weight tile where it is large enough, else through the x tile.
  static constexpr bool kRowsInWeights = kWeightTile >= (size_t)TP * (D + 1);
  static_assert(kRowsInWeights || kPointTile >= (size_t)TP * (D + 1), "write_rows fits");
  static constexpr size_t kVectors = 2 * TP + 2 * TG + kWarps * TP;  // lse2, delta | beta, dS | sums of a pass
};

__device__ __forceinline__ bool tau_ok(float t) { return t > 0.f && t < INFINITY; }
__device__ __forceinline__ float masked_bias(float b) { return b < kMaskedBias ? kMaskedBias : b; }
// The call's first launch writes the status word: one block looks at every temperature.
__device__ __forceinline__ void write_status(bool reset, const float* tau, int H, uint32_t* status) {
  if (!reset || blockIdx.x + blockIdx.y + blockIdx.z != 0) return;
  int bad = 0;
  for (int h = threadIdx.x; h < H; h += blockDim.x) bad |= !tau_ok(tau[h]);
  bad = __syncthreads_or(bad);
  if (threadIdx.x == 0) *status = bad ? kDevBadTau : kDevOk;
}

// ---- staging ---------------------------------------------------------------------------------
// A tile's operands go from memory through registers to shared memory: load() issues all of a
// thread's reads at once, store() lays them out.  The passes load the next tile before the
// second product of the current one (whose register tile is small), so the reads run under it;
// the backward's slot pass, whose three point tiles would spill there, loads them before the
// barrier that ends the previous tile.  Staged four reads of a loop at a time, the FMA pipe was
// 44 to 50% busy (B = 2, N = 65,536, H = 8, d = 32, G = 256, fp32: whole backward with
// statistics 6944 us, 6047 with this and slot_products over halves of the points; the point
// pass 3292 -> 2900, its FMA pipe 55% busy).

// Points [n0, n0 + TP) of head h, to channel-major; rows past N are zero.
template <int D, int NT, typename T>
struct PointRows {
  static constexpr int kV = 16 / sizeof(T), kN = TP * D / (kV * NT);
  uint4 v[kN];
  __device__ __forceinline__ void load(const T* src, int64_t b, int h, int64_t n0, int64_t N, int H) {
    const int64_t n = n0 + threadIdx.x % TP;
    const T* row = src + ((b * N + n) * H + h) * D + threadIdx.x / TP * kV;
#pragma unroll
    for (int i = 0; i < kN; i++)
      v[i] = n < N ? *reinterpret_cast<const uint4*>(row + i * (NT / TP) * kV) : make_uint4(0u, 0u, 0u, 0u);
  }
  __device__ __forceinline__ void store(float* dst) const {
    dst += threadIdx.x / TP * kV * LP + threadIdx.x % TP;
#pragma unroll
    for (int i = 0; i < kN; i++) {
      const uint32_t w[4] = {v[i].x, v[i].y, v[i].z, v[i].w};
      float* d = dst + i * (NT / TP) * kV * LP;
#pragma unroll
      for (int e = 0; e < 4; e++) {
        if (sizeof(T) == 4) {
          d[e * LP] = __uint_as_float(w[e]);
        } else {
          d[2 * e * LP] = __uint_as_float(w[e] << 16);
          d[(2 * e + 1) * LP] = __uint_as_float(w[e] & 0xffff0000u);
        }
      }
    }
  }
};
// Slots [g0, g0 + TG) of W[h] and the bias, scaled on their way to shared memory.  Rows of W
// are G floats: read by fours where G is a multiple of four, else by ones.
template <int D, int TG, int NT>
struct SlotW {
  static constexpr int kN = TG * D / NT;
  static_assert(kN % 4 == 0 && TG <= NT, "whole pieces");
  float v[kN], bias;
  __device__ __forceinline__ void load(const float* W, const float* bs, int h, int G, int g0) {
    W += (int64_t)h * D * G + g0;
    if (G % 4 == 0) {
#pragma unroll
      for (int i = 0; i < kN / 4; i++) {
        const int t = threadIdx.x + i * NT, g = t % (TG / 4) * 4, k = t / (TG / 4);
        const float4 f = g0 + g < G ? *reinterpret_cast<const float4*>(W + (int64_t)k * G + g)
                                    : make_float4(0.f, 0.f, 0.f, 0.f);
        v[4 * i] = f.x, v[4 * i + 1] = f.y, v[4 * i + 2] = f.z, v[4 * i + 3] = f.w;
      }
    } else {
#pragma unroll
      for (int i = 0; i < kN; i++) {
        const int t = threadIdx.x + i * NT, g = t % TG, k = t / TG;
        v[i] = g0 + g < G ? W[(int64_t)k * G + g] : 0.f;
      }
    }
    const int g = g0 + (int)threadIdx.x;
    bias = (int)threadIdx.x < TG && g < G ? bs[(int64_t)h * G + g] : 0.f;
  }
  __device__ __forceinline__ void store(float* dst, float* sB, int G, int g0, float scale) const {
    if (G % 4 == 0) {
#pragma unroll
      for (int i = 0; i < kN / 4; i++) {
        const int t = threadIdx.x + i * NT, g = t % (TG / 4) * 4, k = t / (TG / 4);
        *reinterpret_cast<float4*>(dst + k * (TG + 4) + g) =
            make_float4(v[4 * i] * scale, v[4 * i + 1] * scale, v[4 * i + 2] * scale, v[4 * i + 3] * scale);
      }
    } else {
#pragma unroll
      for (int i = 0; i < kN; i++) {
        const int t = threadIdx.x + i * NT;
        dst[t / TG * (TG + 4) + t % TG] = v[i] * scale;
      }
    }
    if (threadIdx.x < TG) sB[threadIdx.x] = g0 + (int)threadIdx.x < G ? masked_bias(bias * scale) : kLowest;
  }
};
// Token rows [g0, g0 + TG) of t [G][D], to channel-major.
template <int D, int TG, int NT>
struct TokenRows {
  static constexpr int kN = TG * D / (4 * NT);
  static_assert(kN >= 1, "whole pieces");
  float4 v[kN];
  __device__ __forceinline__ void load(const float* t, int G, int g0) {
#pragma unroll
    for (int i = 0; i < kN; i++) {
      const int e = threadIdx.x + i * NT, g = e % TG, c = e / TG * 4;
      v[i] = g0 + g < G ? *reinterpret_cast<const float4*>(t + (int64_t)(g0 + g) * D + c)
                        : make_float4(0.f, 0.f, 0.f, 0.f);
    }
  }
  __device__ __forceinline__ void store(float* dst) const {
#pragma unroll
    for (int i = 0; i < kN; i++) {
      const int e = threadIdx.x + i * NT, g = e % TG, c = e / TG * 4;
      dst[c * (TG + 4) + g] = v[i].x;
      dst[(c + 1) * (TG + 4) + g] = v[i].y;
      dst[(c + 2) * (TG + 4) + g] = v[i].z;
      dst[(c + 3) * (TG + 4) + g] = v[i].w;
    }
  }
};
// One value per point (lse, delta) or slot (dS), by the first threads.
__device__ __forceinline__ float load_one(const float* src, int64_t i, int64_t n, int count) {
  return (int)threadIdx.x < count && i + threadIdx.x < n ? src[i + threadIdx.x] : 0.f;
}
__device__ __forceinline__ void store_lse2(float* dst, float lse, int64_t n0, int64_t N) {
  if (threadIdx.x < TP) dst[threadIdx.x] = n0 + threadIdx.x < N ? lse * kLog2e : kFar;
}

// ---- products --------------------------------------------------------------------------------
__device__ __forceinline__ void ld4(float* v, const float* p) {
  const float4 t = *reinterpret_cast<const float4*>(p);
  v[0] = t.x, v[1] = t.y, v[2] = t.z, v[3] = t.w;
}

// Thread (m = lane >> 2, n = lane & 3) of warp (wr, wc): points wr 64 + 32 q + 4 m + i
// (q < 2, i < 4), slots wc 4 N + 16 q + 4 n + j.  pts and slots already point at the
// thread's first point and slot.
template <int K, int N, int LG>
__device__ __forceinline__ void pair_products(float (&acc)[8][N], const float* pts, const float* slots) {
#pragma unroll 4
  for (int k = 0; k < K; k++) {
    float a[8], b[N];
    ld4(a, pts + k * LP);
    ld4(a + 4, pts + k * LP + 32);
#pragma unroll
    for (int q = 0; q < N / 4; q++) ld4(b + 4 * q, slots + k * LG + 16 * q);
#pragma unroll
    for (int i = 0; i < 8; i++)
#pragma unroll
      for (int j = 0; j < N; j++) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
  }
}
// The thread's points as above with M points (M / 4 runs, 32 apart), channels
// 16 wc + n + 4 j.
// Over the tile's first `left` slots, rounded up to eight (the rest have weight 0).
template <int TG, int M, int N>
__device__ __forceinline__ void point_products(float (&acc)[M][N], const float* wts, const float* slots, int left) {
  const int end = min(TG, left);
#pragma unroll 1
  for (int g0 = 0; g0 < end; g0 += 8) {
#pragma unroll
    for (int g = g0; g < g0 + 8; g += 4) {
      float b[N][4];
#pragma unroll
      for (int j = 0; j < N; j++) ld4(b[j], slots + 4 * j * (TG + 4) + g);
#pragma unroll
      for (int e = 0; e < 4; e++) {
        float a[M];
#pragma unroll
        for (int q = 0; q < M / 4; q++) ld4(a + 4 * q, wts + (g + e) * LP + 32 * q);
#pragma unroll
        for (int i = 0; i < M; i++)
#pragma unroll
          for (int j = 0; j < N; j++) acc[i][j] = fmaf(a[i], b[j][e], acc[i][j]);
      }
    }
  }
}
// Slots m + 8 i, channels wc 4 N + n + 4 j, over the warp's half of the points.  (With the warps
// over slots instead, 4 x 4 outputs a thread, the reads took 1.6 clocks per clock of FMAs
// against 1.1.)
template <int M, int N>
__device__ __forceinline__ void slot_products(float (&acc)[M][N], const float* wts, const float* pts) {
#pragma unroll 2
  for (int p = 0; p < TP / 2; p += 4) {
    float a[M][4], b[N][4];
#pragma unroll
    for (int i = 0; i < M; i++) ld4(a[i], wts + 8 * i * LP + p);
#pragma unroll
    for (int j = 0; j < N; j++) ld4(b[j], pts + 4 * j * LP + p);
#pragma unroll
    for (int e = 0; e < 4; e++)
#pragma unroll
      for (int i = 0; i < M; i++)
#pragma unroll
        for (int j = 0; j < N; j++) acc[i][j] = fmaf(a[i][e], b[j][e], acc[i][j]);
  }
}

// A thread's place in the three products.
template <int D, int TG>
struct Place {
  using C = Tile<D, TG>;
  int m, n;
  int p1, g1, c1;  // pair_products: first point and slot; its warp column
  int p2, c2, w2;  // point_products: first point and channel; its warp column
  int p3, c3;      // slot_products: first point and channel (first slot: m)
  __device__ __forceinline__ Place() {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    m = lane >> 2, n = lane & 3;
    p1 = (warp & 1) * 64 + 4 * m;
    c1 = warp >> 1;
    g1 = c1 * 4 * C::kPairN + 4 * n;
    w2 = warp / C::kPtRows;
    p2 = (warp % C::kPtRows) * 8 * C::kPtM + 4 * m;
    c2 = w2 * 16 + n;
    p3 = (warp & 1) * (TP / 2);
    c3 = (warp >> 1) * 4 * C::kSlN + n;
  }
  // point i (of 8) and slot j (of kPairN) of the thread, counted in the tile
  __device__ __forceinline__ int point(int i) const { return p1 + (i >> 2) * 32 + (i & 3); }
  __device__ __forceinline__ int slot(int j) const { return g1 + (j >> 2) * 16 + (j & 3); }
  // Whether the warp's slots of a tile with `left` slots hold any: the pair_products of a warp
  // whose slots are all past G are left out (a tile of 64 and one of 1 slot take G = 65: deslice
  // at N = 131,072, H = 8, d = 16, fp32 272 us with them and all of point_products, 229 without).
  __device__ __forceinline__ bool live(int left) const { return c1 * 4 * C::kPairN < left; }
};

// The thread's 8 x N weights to the tile [slot][point].
template <int D, int TG, int N>
__device__ __forceinline__ void store_weights(float* wts, const Place<D, TG>& pl, const float (&w)[8][N]) {
#pragma unroll
  for (int j = 0; j < N; j++) {
    float* row = wts + pl.slot(j) * LP + pl.p1;
    *reinterpret_cast<float4*>(row) = make_float4(w[0][j], w[1][j], w[2][j], w[3][j]);
    *reinterpret_cast<float4*>(row + 32) = make_float4(w[4][j], w[5][j], w[6][j], w[7][j]);
  }
}

// The two halves' slot_products, the second added to the first through `stage` (free for the
// block, TG D floats); the threads of the first half (p3 = 0) hold the sum.
template <int D, int TG>
__device__ __forceinline__ void add_halves(float (&acc)[Tile<D, TG>::kSlM][Tile<D, TG>::kSlN], float* stage,
                                           const Place<D, TG>& pl) {
  using C = Tile<D, TG>;
  __syncthreads();
#pragma unroll
  for (int i = 0; i < C::kSlM; i++)
#pragma unroll
    for (int j = 0; j < C::kSlN; j++)
      if (pl.p3 != 0) stage[(pl.m + 8 * i) * D + pl.c3 + 4 * j] = acc[i][j];
  __syncthreads();
#pragma unroll
  for (int i = 0; i < C::kSlM; i++)
#pragma unroll
    for (int j = 0; j < C::kSlN; j++)
      if (pl.p3 == 0) acc[i][j] += stage[(pl.m + 8 * i) * D + pl.c3 + 4 * j];
}

// Sum over the four lanes of a run (lane & 3), in a fixed order; every lane gets it.
__device__ __forceinline__ float run_sum(float v) {
  v += __shfl_xor_sync(0xffffffffu, v, 1);
  v += __shfl_xor_sync(0xffffffffu, v, 2);
  return v;
}

__device__ __forceinline__ void store4(float* p, float a, float b, float c, float d) {
  *reinterpret_cast<float4*>(p) = make_float4(a, b, c, d);
}
__device__ __forceinline__ void store4(__nv_bfloat16* p, float a, float b, float c, float d) {
  const __nv_bfloat162 u = __floats2bfloat162_rn(a, b), v = __floats2bfloat162_rn(c, d);
  *reinterpret_cast<uint2*>(p) =
      make_uint2(*reinterpret_cast<const uint32_t*>(&u), *reinterpret_cast<const uint32_t*>(&v));
}
__device__ __forceinline__ void load4(const float* p, float (&v)[4]) { ld4(v, p); }
__device__ __forceinline__ void load4(const __nv_bfloat16* p, float (&v)[4]) {
  const uint2 t = *reinterpret_cast<const uint2*>(p);
  v[0] = __uint_as_float(t.x << 16), v[1] = __uint_as_float(t.x & 0xffff0000u);
  v[2] = __uint_as_float(t.y << 16), v[3] = __uint_as_float(t.y & 0xffff0000u);
}

// A point_products result times `mul` to rows of the points (plus what is there, with
// `add`), through the tile `stage` (at least TP (D + 1) floats, free for the block) so that
// the rows leave in 16-byte (bf16: 8-byte) pieces.
template <int D, int TG, typename T>
__device__ __forceinline__ void write_rows(const float (&acc)[Tile<D, TG>::kPtM][4], float mul, bool add,
                                           float* stage, const Place<D, TG>& pl, T* dst, int64_t b, int h, int64_t n0,
                                           int64_t N, int H) {
  using C = Tile<D, TG>;
  __syncthreads();
#pragma unroll
  for (int i = 0; i < C::kPtM; i++)
#pragma unroll
    for (int j = 0; j < 4; j++)
      stage[(pl.p2 + (i >> 2) * 32 + (i & 3)) * (D + 1) + pl.c2 + 4 * j] = acc[i][j] * mul;
  __syncthreads();
  for (int i = threadIdx.x; i < TP * (D / 4); i += C::kThreads) {
    const int p = i / (D / 4), c = i % (D / 4) * 4;
    if (n0 + p >= N) continue;
    const float* s = stage + p * (D + 1) + c;
    T* o = dst + ((b * N + n0 + p) * H + h) * D + c;
    float old[4] = {0.f, 0.f, 0.f, 0.f};
    if (add) load4(o, old);
    store4(o, s[0] + old[0], s[1] + old[1], s[2] + old[2], s[3] + old[3]);
  }
  __syncthreads();
}

template <int D, int TG>
__host__ __device__ constexpr size_t tile_bytes(int points, int slots, int weights) {
  using C = Tile<D, TG>;
  return (points * C::kPointTile + slots * C::kSlotTile + weights * C::kWeightTile + C::kVectors) * sizeof(float);
}
template <int D, int TG>
constexpr int resident(int blocks) { return Tile<D, TG>::kThreads == 256 ? 1 : blocks; }
// The statistics and the deslice do little per tile at d = 16 and with the narrow tile: on grids of
// many waves more resident blocks hide its barriers and reads (deslice at N = 131,072, H = 8, fp32:
// d = 16, G = 65 229 us with two blocks, 194 with three; d = 16, G = 16 83 with three, 73 with
// four; d = 32, G = 8 154 with two, 130 with three).  Below three blocks an SM the extra ones only
// pile up on some SMs (N = 4,096, G = 32: d = 32 7.4 us with two, 10.0 with three).
template <int D, int TG>
constexpr int resident_many(int blocks) {
  return D == 16 ? (TG == 32 ? 4 : 3) : D == 32 && TG == 32 ? 3 : resident<D, TG>(blocks);
}

// ---- statistics --------------------------------------------------------------------------------
template <int D, int TG, typename T, int kBlocks>
__global__ void __launch_bounds__(Tile<D, TG>::kThreads, kBlocks)
    k_tile_stats(const T* __restrict__ x, const float* __restrict__ W, const float* __restrict__ bias,
                 const float* __restrict__ tau, float* __restrict__ lse, int64_t N, int H, int G, int reset,
                 uint32_t* status) {
  grid_begin(x, W, bias, tau);
  write_status(reset, tau, H, status);
  using C = Tile<D, TG>;
  constexpr int NT = C::kThreads, NJ = C::kPairN;
  extern __shared__ __align__(16) float sm[];
  float* sx = sm;
  float* sw = sx + C::kPointTile;
  float* sB = sw + C::kSlotTile;
  float2* red = reinterpret_cast<float2*>(sB + TG);  // [warp columns][TP]
  const int64_t bh = blockIdx.y, b = bh / H;
  const int h = (int)(bh % H);
  if (!tau_ok(tau[h])) return;
  const float scale = kLog2e / tau[h];
  const int64_t n0 = (int64_t)blockIdx.x * TP;
  const Place<D, TG> pl;
  PointRows<D, NT, T> xr;
  SlotW<D, TG, NT> wr;
  xr.load(x, b, h, n0, N, H);
  wr.load(W, bias, h, G, 0);
  xr.store(sx);
  // Running (max, sum) of the thread's slots.
  float mx[8], l[8];
#pragma unroll
  for (int i = 0; i < 8; i++) mx[i] = kLowest, l[i] = 0.f;
  for (int g0 = 0; g0 < G; g0 += TG) {
    __syncthreads();
    wr.store(sw, sB, G, g0, scale);
    __syncthreads();
    if (g0 + TG < G) wr.load(W, bias, h, G, g0 + TG);
    float a[8][NJ];
#pragma unroll
    for (int j = 0; j < NJ; j++) {
      const float bj = sB[pl.slot(j)];
#pragma unroll
      for (int i = 0; i < 8; i++) a[i][j] = bj;
    }
    if (!pl.live(G - g0)) continue;
    pair_products<D, NJ, C::LG>(a, sx + pl.p1, sw + pl.g1);
#pragma unroll
    for (int i = 0; i < 8; i++) {
      float mn = mx[i];
#pragma unroll
      for (int j = 0; j < NJ; j++) mn = fmaxf(mn, a[i][j]);
      float s = 0.f;
#pragma unroll
      for (int j = 0; j < NJ; j++) s += exp2f(a[i][j] - mn);
      l[i] = l[i] * exp2f(mx[i] - mn) + s;
      mx[i] = mn;
    }
  }
  // The four lanes of a run, then the warp columns (in order).
#pragma unroll
  for (int i = 0; i < 8; i++) {
#pragma unroll
    for (int d = 1; d <= 2; d <<= 1) {
      const float om = __shfl_xor_sync(0xffffffffu, mx[i], d), ol = __shfl_xor_sync(0xffffffffu, l[i], d);
      const float mn = fmaxf(mx[i], om);
      l[i] = l[i] * exp2f(mx[i] - mn) + ol * exp2f(om - mn);
      mx[i] = mn;
    }
    if (pl.n == 0) red[pl.c1 * TP + pl.point(i)] = make_float2(mx[i], l[i]);
  }
  __syncthreads();
  for (int p = threadIdx.x; p < TP; p += NT) {
    float M = kLowest, L = 0.f;
#pragma unroll
    for (int c = 0; c < C::kWarps / 2; c++) M = fmaxf(M, red[c * TP + p].x);
#pragma unroll
    for (int c = 0; c < C::kWarps / 2; c++) L += red[c * TP + p].y * exp2f(red[c * TP + p].x - M);
    if (n0 + p < N) lse[bh * N + n0 + p] = (M + log2f(L)) * kLn2;
  }
}

// The thread's log2-weights a2 - lse2 of the staged tile of `left` slots.
template <int D, int TG>
__device__ __forceinline__ void log_weights(float (&a)[8][Tile<D, TG>::kPairN], const Place<D, TG>& pl,
                                            const float* sx, const float* sw, const float* sB, const float* sl,
                                            int left) {
  using C = Tile<D, TG>;
#pragma unroll
  for (int j = 0; j < C::kPairN; j++) {
    const float bj = sB[pl.slot(j)];
#pragma unroll
    for (int i = 0; i < 8; i++) a[i][j] = bj;
  }
  if (pl.live(left)) pair_products<D, C::kPairN, C::LG>(a, sx + pl.p1, sw + pl.g1);
#pragma unroll
  for (int i = 0; i < 8; i++) {
    const float l2 = sl[pl.point(i)];
#pragma unroll
    for (int j = 0; j < C::kPairN; j++) a[i][j] -= l2;
  }
}

// ---- slice: slot-owned partials over a split of the points ---------------------------------------
// grid (slot tiles, B*H, P).  part[p][bh][g][0..D] = (U, S).
template <int D, int TG, typename T>
__global__ void __launch_bounds__(Tile<D, TG>::kThreads, resident<D, TG>(2))
    k_tile_slice(const T* __restrict__ x, const T* __restrict__ f, const float* __restrict__ W,
                 const float* __restrict__ bias, const float* __restrict__ tau, const float* __restrict__ lse,
                 float* __restrict__ part, int64_t N, int H, int G, int P, int reset, uint32_t* status) {
  grid_begin(x, f, W, bias, tau, lse);
  write_status(reset, tau, H, status);
  using C = Tile<D, TG>;
  constexpr int NT = C::kThreads, NJ = C::kPairN;
  extern __shared__ __align__(16) float sm[];
  float* sx = sm;
  float* sf = sx + C::kPointTile;
  float* sw = sf + C::kPointTile;
  float* wt = sw + C::kSlotTile;
  float* sl = wt + C::kWeightTile;
  float* sB = sl + TP;
  float* red = sB + TG;  // [2 warp rows][TG]
  const int g0 = blockIdx.x * TG;
  const int64_t bh = blockIdx.y, b = bh / H;
  const int h = (int)(bh % H);
  if (!tau_ok(tau[h])) return;
  const Place<D, TG> pl;
  PointRows<D, NT, T> xr, fr;
  float lr;
  auto load = [&](int64_t t) {
    xr.load(x, b, h, t * TP, N, H);
    fr.load(f, b, h, t * TP, N, H);
    lr = load_one(lse + bh * N, t * TP, N, TP);
  };
  {
    SlotW<D, TG, NT> wr;
    wr.load(W, bias, h, G, g0);
    wr.store(sw, sB, G, g0, kLog2e / tau[h]);
  }
  float U[C::kSlM][C::kSlN], S[NJ];
#pragma unroll
  for (int i = 0; i < C::kSlM; i++)
#pragma unroll
    for (int j = 0; j < C::kSlN; j++) U[i][j] = 0.f;
#pragma unroll
  for (int j = 0; j < NJ; j++) S[j] = 0.f;
  const int64_t tiles = (N + TP - 1) / TP, t0 = tiles * blockIdx.z / P, t1 = tiles * (blockIdx.z + 1) / P;
  if (t0 < t1) load(t0);
  for (int64_t t = t0; t < t1; t++) {
    __syncthreads();
    xr.store(sx);
    fr.store(sf);
    store_lse2(sl, lr, t * TP, N);
    __syncthreads();
    float w[8][NJ];
    log_weights<D, TG>(w, pl, sx, sw, sB, sl, G - g0);
#pragma unroll
    for (int j = 0; j < NJ; j++) {
      float s = 0.f;
#pragma unroll
      for (int i = 0; i < 8; i++) {
        w[i][j] = exp2f(w[i][j]);
        s += w[i][j];
      }
      S[j] += s;
    }
    store_weights<D, TG>(wt, pl, w);
    __syncthreads();
    if (t + 1 < t1) load(t + 1);
    slot_products<C::kSlM, C::kSlN>(U, wt + pl.m * LP + pl.p3, sf + pl.c3 * LP + pl.p3);
  }
  // S: the eight runs of a warp, then its two rows of warps.
#pragma unroll
  for (int j = 0; j < NJ; j++) {
#pragma unroll
    for (int d = 4; d <= 16; d <<= 1) S[j] += __shfl_xor_sync(0xffffffffu, S[j], d);
    if (pl.m == 0) red[(threadIdx.x >> 5 & 1) * TG + pl.slot(j)] = S[j];
  }
  add_halves<D, TG>(U, wt, pl);
  float* o = part + (((int64_t)blockIdx.z * gridDim.y + bh) * G + g0) * (D + 1);
#pragma unroll
  for (int i = 0; i < C::kSlM; i++) {
    const int g = pl.m + 8 * i;
    if (pl.p3 != 0 || g0 + g >= G) continue;
#pragma unroll
    for (int j = 0; j < C::kSlN; j++) o[g * (D + 1) + pl.c3 + 4 * j] = U[i][j];
  }
  for (int g = threadIdx.x; g < TG; g += NT)
    if (g0 + g < G) o[g * (D + 1) + D] = red[g] + red[TG + g];
}

// ---- deslice: point-owned ------------------------------------------------------------------------
template <int D, int TG, typename T, int kBlocks>
__global__ void __launch_bounds__(Tile<D, TG>::kThreads, kBlocks)
    k_tile_deslice(const T* __restrict__ x, const float* __restrict__ W, const float* __restrict__ bias,
                   const float* __restrict__ tau, const float* __restrict__ zp, const float* __restrict__ lse,
                   T* __restrict__ out, int64_t N, int H, int G, int reset, uint32_t* status) {
  grid_begin(x, W, bias, tau, zp, lse);
  write_status(reset, tau, H, status);
  using C = Tile<D, TG>;
  constexpr int NT = C::kThreads, NJ = C::kPairN;
  extern __shared__ __align__(16) float sm[];
  float* sx = sm;
  float* sw = sx + C::kPointTile;
  float* sz = sw + C::kSlotTile;
  float* wt = sz + C::kSlotTile;
  float* sl = wt + C::kWeightTile;
  float* sB = sl + TP;
  const int64_t bh = blockIdx.y, b = bh / H;
  const int h = (int)(bh % H);
  if (!tau_ok(tau[h])) return;
  const float scale = kLog2e / tau[h];
  const int64_t n0 = (int64_t)blockIdx.x * TP;
  const Place<D, TG> pl;
  SlotW<D, TG, NT> wr;
  TokenRows<D, TG, NT> zr;
  auto load = [&](int g0) {
    wr.load(W, bias, h, G, g0);
    zr.load(zp + bh * G * D, G, g0);
  };
  {
    PointRows<D, NT, T> xr;
    xr.load(x, b, h, n0, N, H);
    load(0);
    xr.store(sx);
  }
  store_lse2(sl, load_one(lse + bh * N, n0, N, TP), n0, N);
  float acc[C::kPtM][4];
#pragma unroll
  for (int i = 0; i < C::kPtM; i++)
#pragma unroll
    for (int j = 0; j < 4; j++) acc[i][j] = 0.f;
  for (int g0 = 0; g0 < G; g0 += TG) {
    __syncthreads();
    wr.store(sw, sB, G, g0, scale);
    zr.store(sz);
    __syncthreads();
    float w[8][NJ];
    log_weights<D, TG>(w, pl, sx, sw, sB, sl, G - g0);
#pragma unroll
    for (int i = 0; i < 8; i++)
#pragma unroll
      for (int j = 0; j < NJ; j++) w[i][j] = exp2f(w[i][j]);
    store_weights<D, TG>(wt, pl, w);
    __syncthreads();
    if (g0 + TG < G) load(g0 + TG);
    point_products<TG>(acc, wt + pl.p2, sz + pl.c2 * C::LG, G - g0);
  }
  write_rows<D, TG, T>(acc, 1.f, false, C::kRowsInWeights ? wt : sx, pl, out, b, h, n0, N, H);
}

// ---- backward, point-owned -----------------------------------------------------------------------
// Gradient with respect to the weight of point n at slot g (App. G.1):
//   dw_g = [deslice] dO . z'_g  +  [slice] f . dU_g + dS_g,   delta = sum_g w_g dw_g,
//   da_g = w_g (dw_g - delta).
// MODE 0: the deslice's terms, 1: the slice's, 2: both (their da share the weights, so one
// pass serves both).
// Sweep 1 forms R = sum_g w_g z'_g and dfx = sum_g w_g dU_g, and from them
// delta = dO . R + f . dfx + sum_g w_g dS_g: 3 d products per pair and both parts, where
// summing w_g dw_g takes 4 d.  Sweep 2 forms dx = (1/tau) sum_g da_g W[:,g] and the
// points' terms of the temperature gradient, sum_g da_g (a_g - lse) in base-2 units: with the
// logits centred on lse (exact, since sum_g da_g = 0) they carry no large cancelling parts
// (App. G.2).
template <int D, int TG, typename T, int MODE>
__global__ void __launch_bounds__(Tile<D, TG>::kThreads, resident<D, TG>(2))
    k_tile_bwd_point(const T* __restrict__ x, const T* __restrict__ dO, const T* __restrict__ fx,
                     const float* __restrict__ W, const float* __restrict__ bias, const float* __restrict__ tau,
                     const float* __restrict__ zp, const float* __restrict__ dUS, const float* __restrict__ lse,
                     T* __restrict__ dx, T* __restrict__ dfx, float* __restrict__ delta, float* __restrict__ dt_part,
                     int accumulate, int64_t N, int H, int G, int reset, uint32_t* status) {
  grid_begin(x, dO, fx, W, bias, tau, zp, dUS, lse);
  write_status(reset, tau, H, status);
  using C = Tile<D, TG>;
  constexpr int NT = C::kThreads, NJ = C::kPairN, M2 = C::kPtM;
  constexpr bool kD = MODE != 1, kS = MODE != 0;
  extern __shared__ __align__(16) float sm[];
  float* sx = sm;
  float* sd = sx + C::kPointTile;                         // dO
  float* sf = sd + (kD ? C::kPointTile : 0);              // fx
  float* sw = sf + (kS ? C::kPointTile : 0);
  float* sz = sw + C::kSlotTile;                          // z'
  float* su = sz + (kD ? C::kSlotTile : 0);               // dU
  float* wt = su + (kS ? C::kSlotTile : 0);
  float* sl = wt + C::kWeightTile;
  float* sdl = sl + TP;
  float* sB = sdl + TP;
  float* sS = sB + TG;
  float* red = sS + TG;  // [4][TP]
  const int64_t bh = blockIdx.y, b = bh / H;
  const int h = (int)(bh % H);
  if (!tau_ok(tau[h])) return;
  const float scale = kLog2e / tau[h];
  const int64_t n0 = (int64_t)blockIdx.x * TP;
  const Place<D, TG> pl;
  {
    PointRows<D, NT, T> r;
    r.load(x, b, h, n0, N, H);
    r.store(sx);
    if (kD) r.load(dO, b, h, n0, N, H), r.store(sd);
    if (kS) r.load(fx, b, h, n0, N, H), r.store(sf);
  }
  store_lse2(sl, load_one(lse + bh * N, n0, N, TP), n0, N);
  const float* zb = kD ? zp + bh * G * D : nullptr;
  const float* ub = kS ? dUS + bh * G * D : nullptr;
  const float* sb = kS ? dUS + ((int64_t)gridDim.y * D + bh) * G : nullptr;
  SlotW<D, TG, NT> wr;
  TokenRows<D, TG, NT> zr, ur;
  float sr;
  auto load = [&](int g0) {
    wr.load(W, bias, h, G, g0);
    if (kD) zr.load(zb, G, g0);
    if (kS) ur.load(ub, G, g0), sr = load_one(sb, g0, G, TG);
  };
  auto stage = [&](int g0) {
    __syncthreads();
    wr.store(sw, sB, G, g0, scale);
    if (kD) zr.store(sz);
    if (kS) {
      ur.store(su);
      if (threadIdx.x < TG) sS[threadIdx.x] = sr;
    }
    __syncthreads();
  };
  load(0);
  // Sweep 1: R, dfx, sum_g w dS.
  {
    float R[M2][4], F[M2][4], ws[8];
#pragma unroll
    for (int i = 0; i < M2; i++)
#pragma unroll
      for (int j = 0; j < 4; j++) R[i][j] = 0.f, F[i][j] = 0.f;
#pragma unroll
    for (int i = 0; i < 8; i++) ws[i] = 0.f;
    for (int g0 = 0; g0 < G; g0 += TG) {
      stage(g0);
      float w[8][NJ];
      log_weights<D, TG>(w, pl, sx, sw, sB, sl, G - g0);
#pragma unroll
      for (int j = 0; j < NJ; j++) {
        const float s = kS ? sS[pl.slot(j)] : 0.f;
#pragma unroll
        for (int i = 0; i < 8; i++) {
          w[i][j] = exp2f(w[i][j]);
          if (kS) ws[i] = fmaf(w[i][j], s, ws[i]);
        }
      }
      store_weights<D, TG>(wt, pl, w);
      __syncthreads();
      load(g0 + TG < G ? g0 + TG : 0);  // (the second sweep's first tile at last)
      if (kD) point_products<TG>(R, wt + pl.p2, sz + pl.c2 * C::LG, G - g0);
      if (kS) point_products<TG>(F, wt + pl.p2, su + pl.c2 * C::LG, G - g0);
    }
    // delta: the dot products of the thread's channels, over the run, then the warp
    // columns in order; then the columns' sums of w dS.
#pragma unroll
    for (int i = 0; i < M2; i++) {
      const int p = pl.p2 + (i >> 2) * 32 + (i & 3);
      float v = 0.f;
#pragma unroll
      for (int j = 0; j < 4; j++) {
        if (kD) v = fmaf(sd[(pl.c2 + 4 * j) * LP + p], R[i][j], v);
        if (kS) v = fmaf(sf[(pl.c2 + 4 * j) * LP + p], F[i][j], v);
      }
      v = run_sum(v);
      if (pl.n == 0) red[pl.w2 * TP + p] = v;
    }
    __syncthreads();
    for (int p = threadIdx.x; p < TP; p += NT) {
      float v = red[p];
#pragma unroll
      for (int c = 1; c < C::kPtCols; c++) v += red[c * TP + p];
      sdl[p] = v;
    }
    if (kS) {
      __syncthreads();
#pragma unroll
      for (int i = 0; i < 8; i++) {
        const float v = run_sum(ws[i]);
        if (pl.n == 0) red[pl.c1 * TP + pl.point(i)] = v;
      }
      __syncthreads();
      for (int p = threadIdx.x; p < TP; p += NT) {
        float v = sdl[p];
#pragma unroll
        for (int c = 0; c < C::kWarps / 2; c++) v += red[c * TP + p];
        sdl[p] = v;
      }
      write_rows<D, TG, T>(F, 1.f, false, wt, pl, dfx, b, h, n0, N, H);
    }
    __syncthreads();
    for (int p = threadIdx.x; p < TP; p += NT)
      if (n0 + p < N) delta[bh * N + n0 + p] = sdl[p];
  }
  // Sweep 2: dx and the temperature terms.
  float acc[M2][4], dt = 0.f;
#pragma unroll
  for (int i = 0; i < M2; i++)
#pragma unroll
    for (int j = 0; j < 4; j++) acc[i][j] = 0.f;
  for (int g0 = 0; g0 < G; g0 += TG) {
    stage(g0);
    float a[8][NJ], dw[8][NJ];
    log_weights<D, TG>(a, pl, sx, sw, sB, sl, G - g0);
#pragma unroll
    for (int j = 0; j < NJ; j++) {
      const float s = kS ? sS[pl.slot(j)] : 0.f;
#pragma unroll
      for (int i = 0; i < 8; i++) dw[i][j] = s;
    }
    if (pl.live(G - g0)) {
      if (kD) pair_products<D, NJ, C::LG>(dw, sd + pl.p1, sz + pl.g1);
      if (kS) pair_products<D, NJ, C::LG>(dw, sf + pl.p1, su + pl.g1);
    }
#pragma unroll
    for (int i = 0; i < 8; i++) {
      const float dl = sdl[pl.point(i)];
#pragma unroll
      for (int j = 0; j < NJ; j++) {
        const float da = exp2f(a[i][j]) * (dw[i][j] - dl);
        dt = fmaf(da, a[i][j], dt);
        dw[i][j] = da;
      }
    }
    store_weights<D, TG>(wt, pl, dw);
    __syncthreads();
    if (g0 + TG < G) load(g0 + TG);
    point_products<TG>(acc, wt + pl.p2, sw + pl.c2 * C::LG, G - g0);
  }
  // acc = sum_g da_g W[:,g] log2e/tau; dx = acc ln2.
  write_rows<D, TG, T>(acc, kLn2, accumulate != 0, wt, pl, dx, b, h, n0, N, H);
  // Block sum of the temperature terms (fixed tree order) -> dt_part[bh][block].
  red[threadIdx.x] = dt;
  __syncthreads();
  for (int w = NT / 2; w > 0; w >>= 1) {
    if (threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) dt_part[bh * gridDim.x + blockIdx.x] = red[0] * kLn2;
}

// ---- backward, slot-owned ------------------------------------------------------------------------
// grid (slot tiles, B*H, P); da as in the point pass.
//   dWa_g = sum_n da x_n,  dba_g = sum_n da;  MODE 0 also dz'_g = sum_n w dO_n.
// part[p][bh][g] = (MODE 0: dz' (D)), dWa (D), dba, 0   (un-scaled by 1/tau).
template <int D, int TG, typename T, int MODE>
__global__ void __launch_bounds__(Tile<D, TG>::kThreads, resident<D, TG>(2))
    k_tile_bwd_slot(const T* __restrict__ x, const T* __restrict__ dO, const T* __restrict__ fx,
                    const float* __restrict__ W, const float* __restrict__ bias, const float* __restrict__ tau,
                    const float* __restrict__ zp, const float* __restrict__ dUS, const float* __restrict__ lse,
                    const float* __restrict__ delta, float* __restrict__ part, int64_t N, int H, int G, int P) {
  grid_begin(x, dO, fx, W, bias, tau, zp, dUS, lse, delta);
  using C = Tile<D, TG>;
  constexpr int NT = C::kThreads, NJ = C::kPairN;
  constexpr bool kD = MODE != 1, kS = MODE != 0;
  constexpr int PS = MODE == 0 ? 2 * D + 2 : D + 2, off = MODE == 0 ? D : 0;
  extern __shared__ __align__(16) float sm[];
  float* sx = sm;
  float* sd = sx + C::kPointTile;
  float* sf = sd + (kD ? C::kPointTile : 0);
  float* sw = sf + (kS ? C::kPointTile : 0);
  float* sz = sw + C::kSlotTile;
  float* su = sz + (kD ? C::kSlotTile : 0);
  float* wt = su + (kS ? C::kSlotTile : 0);
  float* sl = wt + C::kWeightTile;
  float* sdl = sl + TP;
  float* sB = sdl + TP;
  float* sS = sB + TG;
  float* red = sS + TG;  // [2 warp rows][TG]
  const int g0 = blockIdx.x * TG;
  const int64_t bh = blockIdx.y, b = bh / H;
  const int h = (int)(bh % H);
  if (!tau_ok(tau[h])) return;
  const Place<D, TG> pl;
  {
    SlotW<D, TG, NT> wr;
    TokenRows<D, TG, NT> tr;
    wr.load(W, bias, h, G, g0);
    wr.store(sw, sB, G, g0, kLog2e / tau[h]);
    if (kD) tr.load(zp + bh * G * D, G, g0), tr.store(sz);
    if (kS) {
      tr.load(dUS + bh * G * D, G, g0), tr.store(su);
      const float v = load_one(dUS + ((int64_t)gridDim.y * D + bh) * G, g0, G, TG);
      if (threadIdx.x < TG) sS[threadIdx.x] = v;
    }
  }
  float dW[C::kSlM][C::kSlN], dZ[C::kSlM][C::kSlN], db[NJ];
#pragma unroll
  for (int i = 0; i < C::kSlM; i++)
#pragma unroll
    for (int j = 0; j < C::kSlN; j++) dW[i][j] = 0.f, dZ[i][j] = 0.f;
#pragma unroll
  for (int j = 0; j < NJ; j++) db[j] = 0.f;
  const int64_t tiles = (N + TP - 1) / TP, t0 = tiles * blockIdx.z / P, t1 = tiles * (blockIdx.z + 1) / P;
  for (int64_t t = t0; t < t1; t++) {
    PointRows<D, NT, T> xr, dr, fr;
    xr.load(x, b, h, t * TP, N, H);
    if (kD) dr.load(dO, b, h, t * TP, N, H);
    if (kS) fr.load(fx, b, h, t * TP, N, H);
    const float lr = load_one(lse + bh * N, t * TP, N, TP), er = load_one(delta + bh * N, t * TP, N, TP);
    __syncthreads();
    xr.store(sx);
    if (kD) dr.store(sd);
    if (kS) fr.store(sf);
    store_lse2(sl, lr, t * TP, N);
    if (threadIdx.x < TP) sdl[threadIdx.x] = er;
    __syncthreads();
    float a[8][NJ], dw[8][NJ];
    log_weights<D, TG>(a, pl, sx, sw, sB, sl, G - g0);
#pragma unroll
    for (int j = 0; j < NJ; j++) {
      const float s = kS ? sS[pl.slot(j)] : 0.f;
#pragma unroll
      for (int i = 0; i < 8; i++) dw[i][j] = s;
    }
    if (pl.live(G - g0)) {
      if (kD) pair_products<D, NJ, C::LG>(dw, sd + pl.p1, sz + pl.g1);
      if (kS) pair_products<D, NJ, C::LG>(dw, sf + pl.p1, su + pl.g1);
    }
#pragma unroll
    for (int i = 0; i < 8; i++) {
      const float dl = sdl[pl.point(i)];
#pragma unroll
      for (int j = 0; j < NJ; j++) {
        a[i][j] = exp2f(a[i][j]);
        dw[i][j] = a[i][j] * (dw[i][j] - dl);
      }
    }
#pragma unroll
    for (int j = 0; j < NJ; j++) {
      float s = 0.f;
#pragma unroll
      for (int i = 0; i < 8; i++) s += dw[i][j];
      db[j] += s;
    }
    store_weights<D, TG>(wt, pl, dw);
    __syncthreads();
    slot_products<C::kSlM, C::kSlN>(dW, wt + pl.m * LP + pl.p3, sx + pl.c3 * LP + pl.p3);
    if (MODE == 0) {
      __syncthreads();
      store_weights<D, TG>(wt, pl, a);
      __syncthreads();
      slot_products<C::kSlM, C::kSlN>(dZ, wt + pl.m * LP + pl.p3, sd + pl.c3 * LP + pl.p3);
    }
  }
#pragma unroll
  for (int j = 0; j < NJ; j++) {
#pragma unroll
    for (int d = 4; d <= 16; d <<= 1) db[j] += __shfl_xor_sync(0xffffffffu, db[j], d);
    if (pl.m == 0) red[(threadIdx.x >> 5 & 1) * TG + pl.slot(j)] = db[j];
  }
  add_halves<D, TG>(dW, wt, pl);
  if (MODE == 0) add_halves<D, TG>(dZ, wt, pl);
  float* o = part + (((int64_t)blockIdx.z * gridDim.y + bh) * G + g0) * PS;
#pragma unroll
  for (int i = 0; i < C::kSlM; i++) {
    const int g = pl.m + 8 * i;
    if (pl.p3 != 0 || g0 + g >= G) continue;
#pragma unroll
    for (int j = 0; j < C::kSlN; j++) {
      if (MODE == 0) o[g * PS + pl.c3 + 4 * j] = dZ[i][j];
      o[g * PS + off + pl.c3 + 4 * j] = dW[i][j];
    }
  }
  for (int g = threadIdx.x; g < TG; g += NT)
    if (g0 + g < G) {
      o[g * PS + off + D] = red[g] + red[TG + g];
      o[g * PS + off + D + 1] = 0.f;  // (the temperature gradient is formed per point)
    }
}

// ---- launches --------------------------------------------------------------------------------------
template <typename K>
cudaError_t allow_smem(K kernel, size_t bytes) {
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}
inline bool many_waves(const Shape& s) { return simt_point_blocks(s) * s.BH() > 3 * num_sms(); }
inline dim3 point_grid(const Shape& s) { return dim3((unsigned)((s.N + TP - 1) / TP), (unsigned)s.BH()); }
template <int TG>
dim3 slot_grid(const Shape& s, int P) {
  return dim3((unsigned)((s.G + TG - 1) / TG), (unsigned)s.BH(), (unsigned)P);
}

// Calls fn with (d, slots per tile) of the shape as compile-time constants.  kNarrow64: d = 64 has
// the narrow tile too (the statistics and the deslice, whose sweeps over the slots are all of
// their work: N = 131,072, H = 8, G = 16, fp32, 348 and 576 us with the wide tile, 158 and 288 with the narrow one).
template <bool kNarrow64 = false, typename Fn>
cudaError_t with_tile(const Shape& s, Fn fn) {
  const bool narrow = simt_tile_slots(s) == 32;
#define FS_TILE(D_)                                                                                    \
  return narrow ? fn(std::integral_constant<int, D_>{}, std::integral_constant<int, 32>{})             \
                : fn(std::integral_constant<int, D_>{}, std::integral_constant<int, 64>{})
  switch (s.d) {
    case 16: FS_TILE(16);
    case 32: FS_TILE(32);
    case 64:
      if constexpr (kNarrow64)
        if (s.G <= 32) return fn(std::integral_constant<int, 64>{}, std::integral_constant<int, 32>{});
      return fn(std::integral_constant<int, 64>{}, std::integral_constant<int, 64>{});
    default: return cudaErrorInvalidValue;
  }
#undef FS_TILE
}

}  // namespace

template <typename T>
cudaError_t SimtTiles<T>::stats(const Shape& s, const T* x, const float* W, const float* bias, const float* tau,
                                float* lse, bool reset, uint32_t* status, cudaStream_t st) {
  return with_tile<true>(s, [&](auto d, auto tg) {
    constexpr int D = decltype(d)::value, TG = decltype(tg)::value;
    constexpr size_t sm = tile_bytes<D, TG>(1, 1, 0);
    const auto k = many_waves(s) ? k_tile_stats<D, TG, T, resident_many<D, TG>(3)> : k_tile_stats<D, TG, T, resident<D, TG>(3)>;
    if (cudaError_t e = allow_smem(k, sm)) return e;
    return launch(k, point_grid(s), dim3(Tile<D, TG>::kThreads), sm, st, x, W, bias, tau, lse, s.N, s.H, s.G, reset,
                  status);
  });
}

template <typename T>
cudaError_t SimtTiles<T>::slice(const Shape& s, int P, const T* x, const T* f, const float* W, const float* bias,
                                const float* tau, const float* lse, float* part, bool reset, uint32_t* status,
                                cudaStream_t st) {
  return with_tile(s, [&](auto d, auto tg) {
    constexpr int D = decltype(d)::value, TG = decltype(tg)::value;
    constexpr size_t sm = tile_bytes<D, TG>(2, 1, 1);
    const auto k = k_tile_slice<D, TG, T>;
    if (cudaError_t e = allow_smem(k, sm)) return e;
    return launch(k, slot_grid<TG>(s, P), dim3(Tile<D, TG>::kThreads), sm, st, x, f, W, bias, tau, lse, part, s.N, s.H,
                  s.G, P, reset, status);
  });
}

template <typename T>
cudaError_t SimtTiles<T>::deslice(const Shape& s, const T* x, const float* W, const float* bias, const float* tau,
                                  const float* zp, const float* lse, T* out, bool reset, uint32_t* status,
                                  cudaStream_t st) {
  return with_tile<true>(s, [&](auto d, auto tg) {
    constexpr int D = decltype(d)::value, TG = decltype(tg)::value;
    constexpr size_t sm = tile_bytes<D, TG>(1, 2, 1);
    const auto k =
        many_waves(s) ? k_tile_deslice<D, TG, T, resident_many<D, TG>(2)> : k_tile_deslice<D, TG, T, resident<D, TG>(2)>;
    if (cudaError_t e = allow_smem(k, sm)) return e;
    return launch(k, point_grid(s), dim3(Tile<D, TG>::kThreads), sm, st, x, W, bias, tau, zp, lse, out, s.N, s.H, s.G,
                  reset, status);
  });
}

template <typename T>
cudaError_t SimtTiles<T>::backward(const Shape& s, int mode, int P, const T* x, const T* dO, const T* fx,
                                   const float* W, const float* bias, const float* tau, const float* zp,
                                   const float* dUS, const float* lse, T* dx, T* dfx, float* delta, float* dt_part,
                                   float* part, int accumulate, bool reset, uint32_t* status, cudaStream_t st) {
  return with_tile(s, [&](auto d, auto tg) {
    constexpr int D = decltype(d)::value, TG = decltype(tg)::value, NT = Tile<D, TG>::kThreads;
    auto run = [&](auto m) -> cudaError_t {
      constexpr int MODE = decltype(m)::value, V = MODE == 2 ? 3 : 2;
      constexpr size_t sm = tile_bytes<D, TG>(V, V, 1);
      const auto kp = k_tile_bwd_point<D, TG, T, MODE>;
      if (cudaError_t e = allow_smem(kp, sm)) return e;
      if (cudaError_t e = launch(kp, point_grid(s), dim3(NT), sm, st, x, dO, fx, W, bias, tau, zp, dUS, lse, dx, dfx,
                                 delta, dt_part, accumulate, s.N, s.H, s.G, reset, status))
        return e;
      const auto ks = k_tile_bwd_slot<D, TG, T, MODE>;
      if (cudaError_t e = allow_smem(ks, sm)) return e;
      return launch(ks, slot_grid<TG>(s, P), dim3(NT), sm, st, x, dO, fx, W, bias, tau, zp, dUS, lse, delta, part, s.N,
                    s.H, s.G, P);
    };
    if (mode == 0) return run(std::integral_constant<int, 0>{});
    if (mode == 1) return run(std::integral_constant<int, 1>{});
    return run(std::integral_constant<int, 2>{});
  });
}

}  // namespace fs
