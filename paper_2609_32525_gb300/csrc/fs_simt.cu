// SIMT path: dispatch of the tiled fp32 passes (fs_simt_tiles.cuh), which serve every shape
// the tensor-core kernels do not cover (d != 32, G above their limits, small fp32
// problems, the backward of fp32 inputs), and the small fp32 kernels that every path
// shares: the fixed-order reductions, the mixes and their backward.  No float atomics
// anywhere.
#include "fs_launch.h"
#include "fs_simt_tiles.h"

#include <cuda_bf16.h>

namespace fs {
namespace {

// Fixed-order sum of the P partials [P, BHG, D+1], then (optionally) the
// normalisation.  The sum over splits runs in split order.  Partials hold Gs >= G
// slot rows per (b, h) (the tensor-core path pads G to whole 128-slot blocks);
// only the first G are reduced.
__global__ void k_reduce_tokens(const float* __restrict__ part, int P, int64_t BH, int G, int Gs, int D,
                                float* __restrict__ tokens, float* __restrict__ wsum, int finalize,
                                float eps) {
  grid_begin(part);
  // One warp per output row bh * G + g; lane l sums columns l, l + 32, l + 64 (<= D)
  // of its partial row over the splits, loads four splits ahead.
  const int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (i >= BH * G) return;  // whole warps
  const int64_t row = (i / G) * Gs + i % G;  // its partial row
  const int64_t stride = BH * Gs * (D + 1);
  const float* src = part + row * (D + 1);
  float v[3] = {0.f, 0.f, 0.f};
#pragma unroll
  for (int j = 0; j < 3; j++) {
    const int c = lane + 32 * j;
    if (c > D) continue;
    int p = 0;
    for (; p + 4 <= P; p += 4) {
      const float a0 = src[(int64_t)p * stride + c], a1 = src[(int64_t)(p + 1) * stride + c];
      const float a2 = src[(int64_t)(p + 2) * stride + c], a3 = src[(int64_t)(p + 3) * stride + c];
      v[j] = (((v[j] + a0) + a1) + a2) + a3;
    }
    for (; p < P; p++) v[j] += src[(int64_t)p * stride + c];
  }
  const int jS = D >> 5;  // column D (the weight sum) is lane D % 32's entry jS
  const float S = __shfl_sync(0xffffffffu, jS == 0 ? v[0] : (jS == 1 ? v[1] : v[2]), D & 31);
#pragma unroll
  for (int j = 0; j < 3; j++) {
    const int c = lane + 32 * j;
    if (c < D)
      tokens[i * D + c] = finalize ? v[j] / (S + eps) : v[j];
    else if (c == D)
      wsum[i] = v[j];
  }
}

__global__ void k_finalize(float* __restrict__ tokens, const float* __restrict__ wsum, int64_t BHG,
                           int D, float eps) {
  grid_begin(tokens, wsum);
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= BHG * D) return;
  tokens[i] = tokens[i] / (wsum[i / D] + eps);
}

// ---- mix and its backward ------------------------------------------------------------
// out[bh][g][c] = sum_k A_h(g, k) in[bh][k][c] per (b, h), with A_h = M[h] (the mix,
// z' = M z) or A_h = M[h]^T (its backward, dz = M^T dz').
//
// A block of 8 warps owns a tile of 16 rows g x 32 channels and sweeps k in chunks of
// 64.  A and `in` chunks are staged in shared memory by cp.async, three chunks deep,
// so that two chunks' loads are in flight while one is multiplied.  Warp w takes k
// = 8w .. 8w + 7 of every chunk; each lane keeps a 4 x 4 register tile (4 rows g, 4
// channels), so that two 16-byte shared loads feed 16 FMAs.  The eight warps'
// partial sums are added at the end in warp order: the sum over k has a fixed order.
// kVec: G % 4 == 0, so rows of M move as 16-byte pieces; otherwise as 4-byte words.
constexpr int kMixTG = 16, kMixTC = 32, kMixKC = 64, kMixStages = 3;
// A tile: g-major [16][64 + 4] for the mix (the pad puts the four rows a lane reads,
// g = q, q + 4, q + 8, q + 12, on different banks); k-major [64][16] for the transpose,
// as M[k][g] lies in memory.
template <bool kTrans>
__host__ __device__ constexpr int mix_a_words() { return kTrans ? kMixKC * kMixTG : kMixTG * (kMixKC + 4); }

__device__ __forceinline__ void cp_async16(float* dst, const float* src, bool valid) {
  const unsigned d = static_cast<unsigned>(__cvta_generic_to_shared(dst));
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(d), "l"(src), "r"(valid ? 16 : 0) : "memory");
}
__device__ __forceinline__ void cp_async4(float* dst, const float* src, bool valid) {
  const unsigned d = static_cast<unsigned>(__cvta_generic_to_shared(dst));
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;\n" ::"r"(d), "l"(src), "r"(valid ? 4 : 0) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory"); }

template <bool kTrans>
constexpr int mix_words() { return kMixStages * (mix_a_words<kTrans>() + kMixKC * kMixTC); }

// Tile (gx, bh, cx) of the product, with mix_words() floats of shared memory.
template <bool kTrans, bool kVec>
__device__ __forceinline__ void mix_tile(float* sm, const float* __restrict__ M, const float* __restrict__ in,
                                         float* __restrict__ out, int H, int G, int D, int gx, int64_t bh, int cx) {
  constexpr int TG = kMixTG, TC = kMixTC, KC = kMixKC, S = kMixStages;
  constexpr int AW = mix_a_words<kTrans>(), BW = KC * TC, SW = AW + BW;
  const int h = (int)(bh % H);
  const int g0 = gx * TG, c0 = cx * TC;
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  const float* Mh = M + (int64_t)h * G * G;
  const float* X = in + bh * (int64_t)G * D;
  const int nch = (G + KC - 1) / KC;

  // Stage chunk `ch` (k = ch * KC ...) into buffer `buf`; out-of-range words are zero-filled.
  auto issue = [&](int ch, int buf) {
    if (ch < nch) {
      const int k0 = ch * KC;
      float* sa = sm + buf * SW;
      float* sb = sa + AW;
      if (kVec) {
        if (kTrans) {  // A(g, k) = M[k][g]: row k, 4 consecutive g
          const int k = t >> 2, gg = (t & 3) * 4;
          const bool v = k0 + k < G && g0 + gg < G;
          cp_async16(sa + k * TG + gg, v ? Mh + (int64_t)(k0 + k) * G + g0 + gg : Mh, v);
        } else {  // A(g, k) = M[g][k]: row g, 4 consecutive k
          const int g = t >> 4, kk = (t & 15) * 4;
          const bool v = g0 + g < G && k0 + kk < G;
          cp_async16(sa + g * (KC + 4) + kk, v ? Mh + (int64_t)(g0 + g) * G + k0 + kk : Mh, v);
        }
      } else {
#pragma unroll
        for (int r = 0; r < 4; r++) {
          const int e = t + 256 * r;
          if (kTrans) {
            const int k = e / TG, gg = e % TG;
            const bool v = k0 + k < G && g0 + gg < G;
            cp_async4(sa + k * TG + gg, v ? Mh + (int64_t)(k0 + k) * G + g0 + gg : Mh, v);
          } else {
            const int g = e / KC, kk = e % KC;
            const bool v = g0 + g < G && k0 + kk < G;
            cp_async4(sa + g * (KC + 4) + kk, v ? Mh + (int64_t)(g0 + g) * G + k0 + kk : Mh, v);
          }
        }
      }
#pragma unroll
      for (int r = 0; r < 2; r++) {  // `in` rows k, 4 consecutive channels (D % 4 == 0)
        const int e = t + 256 * r, k = e >> 3, cc = (e & 7) * 4;
        const bool v = k0 + k < G && c0 + cc < D;
        cp_async16(sb + k * TC + cc, v ? X + (int64_t)(k0 + k) * D + c0 + cc : X, v);
      }
    }
    cp_async_commit();
  };

  // Lane (gq, cq): channels 4cq .. 4cq + 3; rows g = gq + 4i (mix) or 4gq + i (transpose).
  const int gq = lane >> 3, cq = lane & 7;
  float acc[4][4] = {};
#pragma unroll
  for (int st = 0; st < S - 1; st++) issue(st, st);
  for (int ch = 0; ch < nch; ch++) {
    cp_async_wait<S - 2>();
    __syncthreads();  // chunk ch is visible; every warp is done with chunk ch - 1's buffer
    issue(ch + S - 1, (ch + S - 1) % S);
    const float* sa = sm + (ch % S) * SW;
    const float* sb = sa + AW;
    if (kTrans) {
#pragma unroll
      for (int kk = 0; kk < 8; kk++) {
        const int k = warp * 8 + kk;
        const float4 a = *reinterpret_cast<const float4*>(sa + k * TG + 4 * gq);
        const float4 b = *reinterpret_cast<const float4*>(sb + k * TC + 4 * cq);
        const float av[4] = {a.x, a.y, a.z, a.w}, bv[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
        for (int i = 0; i < 4; i++)
#pragma unroll
          for (int j = 0; j < 4; j++) acc[i][j] = fmaf(av[i], bv[j], acc[i][j]);
      }
    } else {
#pragma unroll
      for (int half = 0; half < 2; half++) {
        const int kb = warp * 8 + half * 4;
        float av[4][4], bv[4][4];
#pragma unroll
        for (int i = 0; i < 4; i++) {
          const float4 a = *reinterpret_cast<const float4*>(sa + (gq + 4 * i) * (KC + 4) + kb);
          av[i][0] = a.x; av[i][1] = a.y; av[i][2] = a.z; av[i][3] = a.w;
        }
#pragma unroll
        for (int kk = 0; kk < 4; kk++) {
          const float4 b = *reinterpret_cast<const float4*>(sb + (kb + kk) * TC + 4 * cq);
          bv[kk][0] = b.x; bv[kk][1] = b.y; bv[kk][2] = b.z; bv[kk][3] = b.w;
        }
#pragma unroll
        for (int kk = 0; kk < 4; kk++)
#pragma unroll
          for (int i = 0; i < 4; i++)
#pragma unroll
            for (int j = 0; j < 4; j++) acc[i][j] = fmaf(av[i][kk], bv[kk][j], acc[i][j]);
      }
    }
  }
  cp_async_wait<0>();
  __syncthreads();  // the staging buffers become the eight warps' partial tiles
  float* red = sm;  // [8][TG][TC]
#pragma unroll
  for (int i = 0; i < 4; i++) {
    const int g = kTrans ? 4 * gq + i : gq + 4 * i;
    *reinterpret_cast<float4*>(red + (warp * TG + g) * TC + 4 * cq) = make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
  }
  __syncthreads();
#pragma unroll
  for (int r = 0; r < 2; r++) {
    const int o = t + 256 * r, g = o / TC, c = o % TC;
    float v = 0.f;
#pragma unroll
    for (int w = 0; w < 8; w++) v += red[(w * TG + g) * TC + c];
    if (g0 + g < G && c0 + c < D) out[(bh * G + g0 + g) * (int64_t)D + c0 + c] = v;
  }
}
template <bool kTrans, bool kVec>
__global__ void __launch_bounds__(256) k_mix_tiled(const float* __restrict__ M, const float* __restrict__ in,
                                                   float* __restrict__ out, int H, int G, int D) {
  grid_begin(M, in);
  __shared__ __align__(16) float sm[mix_words<kTrans>()];
  mix_tile<kTrans, kVec>(sm, M, in, out, H, G, D, blockIdx.x, blockIdx.y, blockIdx.z);
}
static_assert(8 * kMixTG * kMixTC <= kMixStages * (kMixKC * kMixTC + kMixTG * (kMixKC + 4)),
              "the partial tiles fit in the staging buffers");

// Per-token channel map (the attention-free core): out[bh][g][c] = sum_k A(c, k)
// in[bh][g][k], with A = Wc[h] (forward) or Wc[h]^T (its token backward); one
// thread per output word, the sum over k in a fixed order.
template <bool kTrans>
__global__ void k_mix_channels(const float* __restrict__ Wc, const float* __restrict__ in, float* __restrict__ out,
                               int64_t BHG, int H, int G, int D) {
  grid_begin(Wc, in);
  const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= BHG * D) return;
  const int c = (int)(idx % D);
  const int64_t t = idx / D;  // token bh * G + g
  const int h = (int)((t / G) % H);
  const float* A = Wc + (int64_t)h * D * D;
  const float* z = in + t * D;
  float acc = 0.f;
  for (int k = 0; k < D; k++) acc = fmaf(kTrans ? A[(int64_t)k * D + c] : A[(int64_t)c * D + k], z[k], acc);
  out[idx] = acc;
}

// dWc[h][c][k] = sum over b and g of dzp[b,h,g,c] z[b,h,g,k] (fixed order: b, then g).
__global__ void k_mix_channels_dW(const float* __restrict__ z, const float* __restrict__ dzp, float* __restrict__ dWc,
                                  int64_t B, int H, int G, int D) {
  grid_begin(z, dzp);
  const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (int64_t)H * D * D) return;
  const int k = (int)(idx % D), c = (int)((idx / D) % D), h = (int)(idx / ((int64_t)D * D));
  float acc = 0.f;
  for (int64_t b = 0; b < B; b++) {
    const int64_t base = (b * H + h) * (int64_t)G * D;
    for (int g = 0; g < G; g++) acc = fmaf(dzp[base + (int64_t)g * D + c], z[base + (int64_t)g * D + k], acc);
  }
  dWc[idx] = acc;
}

// dM[h][g][k] = sum_b sum_c dzp[b,h,g,c] z[b,h,k,c]: per head a G x G product with
// K = B*D, tiled 64 x 64 per block (16 x 16 threads, 4 x 4 outputs each), the two
// operand tiles staged in shared memory 16 channels at a time; the sum runs over
// b, then c, in a fixed order.
constexpr int kDmT = 64, kDmKC = 16;
constexpr int kDmWords = 2 * kDmKC * (kDmT + 1);
__device__ __forceinline__ void dM_tile(float* sm, const float* __restrict__ z, const float* __restrict__ dzp,
                                        float* __restrict__ dM, int64_t B, int H, int G, int D, int kx, int gx,
                                        int h) {
  constexpr int T = kDmT, KC = kDmKC;
  float(*sa)[T + 1] = reinterpret_cast<float(*)[T + 1]>(sm);
  float(*sb)[T + 1] = sa + KC;
  const int g0 = gx * T, k0 = kx * T;
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  float acc[4][4] = {};
  for (int64_t b = 0; b < B; b++) {
    const float* A = dzp + (b * H + h) * (int64_t)G * D;
    const float* Z = z + (b * H + h) * (int64_t)G * D;
    for (int c0 = 0; c0 < D; c0 += KC) {
      __syncthreads();
      for (int i = threadIdx.x; i < T * KC; i += 256) {
        const int r = i / KC, c = i % KC;
        sa[c][r] = (g0 + r < G && c0 + c < D) ? A[(int64_t)(g0 + r) * D + c0 + c] : 0.f;
        sb[c][r] = (k0 + r < G && c0 + c < D) ? Z[(int64_t)(k0 + r) * D + c0 + c] : 0.f;
      }
      __syncthreads();
#pragma unroll
      for (int c = 0; c < KC; c++) {
        float av[4], bv[4];
#pragma unroll
        for (int i = 0; i < 4; i++) {
          av[i] = sa[c][ty + 16 * i];
          bv[i] = sb[c][tx + 16 * i];
        }
#pragma unroll
        for (int i = 0; i < 4; i++)
#pragma unroll
          for (int j = 0; j < 4; j++) acc[i][j] = fmaf(av[i], bv[j], acc[i][j]);
      }
    }
  }
#pragma unroll
  for (int i = 0; i < 4; i++) {
    const int g = g0 + ty + 16 * i;
    if (g >= G) continue;
#pragma unroll
    for (int j = 0; j < 4; j++) {
      const int k = k0 + tx + 16 * j;
      if (k < G) dM[((int64_t)h * G + g) * G + k] = acc[i][j];
    }
  }
}

__global__ void __launch_bounds__(256) k_mix_bwd_dM(const float* __restrict__ z, const float* __restrict__ dzp,
                                                    float* __restrict__ dM, int64_t B, int H, int G, int D) {
  grid_begin(z, dzp);
  __shared__ float sm[kDmWords];
  dM_tile(sm, z, dzp, dM, B, H, G, D, blockIdx.x, blockIdx.y, blockIdx.z);
}

// Both halves of the mix backward in one launch: blocks [0, nx * BH * nc) the tiles of
// dz = M^T dz' (gx fastest, then bh), the rest dM's.
template <bool kVec>
__global__ void __launch_bounds__(256) k_mix_bwd(const float* __restrict__ M, const float* __restrict__ z,
                                                 const float* __restrict__ dzp, float* __restrict__ dz,
                                                 float* __restrict__ dM, int64_t B, int H, int G, int D, int nx,
                                                 int nc) {
  grid_begin(M, z, dzp);
  constexpr int kWords = mix_words<true>() > kDmWords ? mix_words<true>() : kDmWords;
  __shared__ __align__(16) float sm[kWords];
  const int64_t n = (int64_t)nx * B * H * nc;
  int64_t i = blockIdx.x;
  if (i < n) {
    const int gx = (int)(i % nx);
    i /= nx;
    mix_tile<true, kVec>(sm, M, dzp, dz, H, G, D, gx, i % (B * H), (int)(i / (B * H)));
    return;
  }
  i -= n;
  const int nt = (G + kDmT - 1) / kDmT;
  dM_tile(sm, z, dzp, dM, B, H, G, D, (int)(i % nt), (int)((i / nt) % nt), (int)(i / ((int64_t)nt * nt)));
}

// Token-gradient prep for the slice backward: dU = dz_g/(S_g+eps) as rows [bh][g][D], then
// dS = -(dz_g.z_g)/(S_g+eps) as [bh][g], so that both read in 16-byte pieces.  A warp
// per slot row (a thread per row read 32-word rows word by word: 20 us at 2,048 rows, 5 us
// this way).
__global__ void __launch_bounds__(256) k_slice_bwd_prep(const float* __restrict__ z, const float* __restrict__ wsum,
                                                        const float* __restrict__ dz, float* __restrict__ dUS,
                                                        int64_t BHG, int D, float eps) {
  grid_begin(z, wsum, dz);
  const int64_t i = ((int64_t)blockIdx.x * 256 + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (i >= BHG) return;  // whole warps
  const float den = wsum[i] + eps;
  float s = 0.f;
  for (int c = lane; c < D; c += 32) {
    const float g = dz[i * D + c];
    dUS[i * D + c] = g / den;
    s = fmaf(g, z[i * D + c], s);
  }
#pragma unroll
  for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane == 0) dUS[BHG * D + i] = -s / den;
}

// Fixed-order reduction of slot-owned backward partials over (b, p), one thread
// per output word (consecutive threads read consecutive words of a partial row):
//   k_reduce_bwd_params: dW[h][k][g], db[h][g] (written, or added), sums over b then p;
//   k_reduce_bwd_tokens: d_tokens_mixed[b][h][g][c], sums over p.
// The temperature gradient is reduced separately, from its own partials.
__device__ __forceinline__ void reduce_params(int64_t idx, const float* __restrict__ part, int P, int64_t B, int H,
                                              int G, int Gs, int D, int PS, int off, const float* __restrict__ tau,
                                              float* __restrict__ dW, float* __restrict__ db, int accumulate) {
  if (idx >= (int64_t)H * G * (D + 1)) return;
  const int k = (int)(idx % (D + 1));
  const int64_t hg = idx / (D + 1);
  const int h = (int)(hg / G), g = (int)(hg % G);
  const int64_t BH = B * H;
  float s = 0.f;
  for (int64_t b = 0; b < B; b++) {
    const float* src = part + ((b * H + h) * Gs + g) * PS + off + k;
#pragma unroll 4
    for (int p = 0; p < P; p++) s += src[(int64_t)p * BH * Gs * PS];
  }
  s *= 1.f / tau[h];
  if (k < D) {
    const int64_t o = ((int64_t)h * D + k) * G + g;
    dW[o] = (accumulate ? dW[o] : 0.f) + s;
  } else {
    db[hg] = (accumulate ? db[hg] : 0.f) + s;
  }
}
__device__ __forceinline__ void reduce_dzp(int64_t idx, const float* __restrict__ part, int P, int64_t BH, int G,
                                           int Gs, int D, int PS, float* __restrict__ dzp) {
  if (idx >= BH * G * D) return;
  const int c = (int)(idx % D);
  const int64_t i = idx / D;                  // output row bh * G + g
  const int64_t row = (i / G) * Gs + i % G;  // its partial row
  float s = 0.f;
#pragma unroll 4
  for (int p = 0; p < P; p++) s += part[((int64_t)p * BH * Gs + row) * PS + c];
  dzp[idx] = s;
}
// dtau[h] (+)= -(1/tau_h) * sum over batches and point blocks of the block sums of
// sum_g da (a - lse) (fixed order: strided per thread, then a tree).  256 threads.
__device__ __forceinline__ void reduce_dtau(int h, const float* __restrict__ dt_part, int64_t B, int H, int64_t nblk,
                                            const float* __restrict__ tau, float* __restrict__ dtau, int accumulate) {
  __shared__ float s[256];
  float v = 0.f;
  for (int64_t b = 0; b < B; b++)
    for (int64_t i = threadIdx.x; i < nblk; i += 256) v += dt_part[(b * H + h) * nblk + i];
  s[threadIdx.x] = v;
  __syncthreads();
  for (int w = 128; w > 0; w >>= 1) {
    if (threadIdx.x < w) s[threadIdx.x] += s[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) dtau[h] = (accumulate ? dtau[h] : 0.f) - s[0] / tau[h];
}

__global__ void __launch_bounds__(256) k_reduce_bwd_params(const float* part, int P, int64_t B, int H, int G, int Gs,
                                                           int D, int PS, int off, const float* tau, float* dW,
                                                           float* db, int accumulate) {
  grid_begin(part, tau);
  reduce_params((int64_t)blockIdx.x * 256 + threadIdx.x, part, P, B, H, G, Gs, D, PS, off, tau, dW, db, accumulate);
}
__global__ void __launch_bounds__(256) k_reduce_bwd_tokens(const float* part, int P, int64_t BH, int G, int Gs, int D,
                                                           int PS, float* dzp) {
  grid_begin(part);
  reduce_dzp((int64_t)blockIdx.x * 256 + threadIdx.x, part, P, BH, G, Gs, D, PS, dzp);
}
__global__ void __launch_bounds__(256) k_reduce_dtau(const float* dt_part, int64_t B, int H, int64_t nblk,
                                                     const float* tau, float* dtau, int accumulate) {
  grid_begin(dt_part, tau);
  reduce_dtau(blockIdx.x, dt_part, B, H, nblk, tau, dtau, accumulate);
}
// All of a backward call's reductions in one launch: blocks [0, n_par) dW and dbias,
// [n_par, n_par + H) dtau, the rest d z' (dzp may be null).
__global__ void __launch_bounds__(256) k_reduce_bwd(const float* part, int P, int64_t B, int H, int G, int Gs, int D,
                                                    int PS, const float* tau, float* dzp, float* dW, float* db,
                                                    float* dtau, const float* dt_part, int64_t nblk, int accumulate,
                                                    int64_t n_par) {
  grid_begin(part, tau, dt_part);
  int64_t blk = blockIdx.x;
  if (blk < n_par)
    return reduce_params(blk * 256 + threadIdx.x, part, P, B, H, G, Gs, D, PS, dzp ? D : 0, tau, dW, db, accumulate);
  blk -= n_par;
  if (blk < H) return reduce_dtau((int)blk, dt_part, B, H, nblk, tau, dtau, accumulate);
  reduce_dzp((blk - H) * 256 + threadIdx.x, part, P, B * H, G, Gs, D, PS, dzp);
}

}  // namespace

cudaError_t simt_reduce_bwd(const Shape& s, int P, const float* part, int Gs, int PS, int has_dzp, const float* tau,
                            float* dzp, float* dW, float* db, float* dtau, const float* dt_part, int64_t nblk,
                            int accumulate, cudaStream_t st) {
  const int64_t nw = (int64_t)s.H * s.G * (s.d + 1);
  cudaError_t e = launch(k_reduce_bwd_params, dim3((unsigned)((nw + 255) / 256)), dim3(256), 0, st, part, P, s.B, s.H,
                         s.G, Gs, s.d, PS, has_dzp ? s.d : 0, tau, dW, db, accumulate);
  if (e != cudaSuccess) return e;
  if (has_dzp) {
    const int64_t BHG = s.BH() * s.G;
    if ((e = launch(k_reduce_bwd_tokens, dim3((unsigned)((BHG * s.d + 255) / 256)), dim3(256), 0, st, part, P, s.BH(),
                    s.G, Gs, s.d, PS, dzp)) != cudaSuccess) return e;
  }
  return launch(k_reduce_dtau, dim3(s.H), dim3(256), 0, st, dt_part, s.B, s.H, nblk, tau, dtau, accumulate);
}

// The one-launch forms of the reductions and of the mix backward serve the tensor-core calls, whose
// chains of launches they shorten; the SIMT calls and fs_mix_bwd still launch the parts one by one.
cudaError_t reduce_bwd(const Shape& s, int P, const float* part, int Gs, int PS, const float* tau, float* dzp,
                       float* dW, float* db, float* dtau, const float* dt_part, int64_t nblk, int accumulate,
                       cudaStream_t st) {
  const int64_t n_par = ((int64_t)s.H * s.G * (s.d + 1) + 255) / 256;
  const int64_t n = n_par + s.H + (dzp ? (s.BH() * s.G * s.d + 255) / 256 : 0);
  return launch(k_reduce_bwd, dim3((unsigned)n), dim3(256), 0, st, part, P, s.B, s.H, s.G, Gs, s.d, PS, tau, dzp, dW,
                db, dtau, dt_part, nblk, accumulate, n_par);
}

cudaError_t mix_bwd(const Shape& s, const float* M, const float* z, const float* dzp, float* dz, float* dM,
                    cudaStream_t st) {
  const int nx = (s.G + kMixTG - 1) / kMixTG, nc = (s.d + kMixTC - 1) / kMixTC, nt = (s.G + kDmT - 1) / kDmT;
  const int64_t n = (int64_t)nx * s.BH() * nc + (int64_t)nt * nt * s.H;
  return launch(s.G % 4 == 0 ? k_mix_bwd<true> : k_mix_bwd<false>, dim3((unsigned)n), dim3(256), 0, st, M, z, dzp, dz,
                dM, s.B, s.H, s.G, s.d, nx, nc);
}

cudaError_t simt_reduce_dzp(const Shape& s, int P, const float* part, int Gs, int PS, float* dzp, cudaStream_t st) {
  const int64_t BHG = s.BH() * s.G;
  return launch(k_reduce_bwd_tokens, dim3((unsigned)((BHG * s.d + 255) / 256)), dim3(256), 0, st, part, P, s.BH(), s.G,
                Gs, s.d, PS, dzp);
}

cudaError_t simt_slice_bwd_prep(const Shape& s, const float* z, const float* wsum, const float* dz, float* dUS,
                                cudaStream_t st) {
  const int64_t BHG = s.BH() * s.G;
  return launch(k_slice_bwd_prep, dim3((unsigned)((BHG + 7) / 8)), dim3(256), 0, st, z, wsum, dz, dUS, BHG, s.d, s.eps);
}

int64_t simt_point_blocks(const Shape& s) { return (s.N + kSimtTP - 1) / kSimtTP; }

// Calls fn with a pointer of the shape's point type.
#define FS_DISPATCH(s, FN, ...) \
  ((s).dtype == FS_BF16 ? FN<__nv_bfloat16>(__VA_ARGS__) : FN<float>(__VA_ARGS__))

namespace {

template <typename T>
const T* in(const void* p) { return static_cast<const T*>(p); }
template <typename T>
T* out(void* p) { return static_cast<T*>(p); }

template <typename T>
cudaError_t launch_stats(const Shape& s, const void* x, const float* W, const float* bias, const float* tau,
                         float* lse, bool reset, uint32_t* status, cudaStream_t st) {
  return SimtTiles<T>::stats(s, in<T>(x), W, bias, tau, lse, reset, status, st);
}
template <typename T>
cudaError_t launch_slice(const Shape& s, int P, const void* x, const void* f, const float* W, const float* bias,
                         const float* tau, const float* lse, float* part, bool reset, uint32_t* status, cudaStream_t st) {
  return SimtTiles<T>::slice(s, P, in<T>(x), in<T>(f), W, bias, tau, lse, part, reset, status, st);
}
template <typename T>
cudaError_t launch_deslice(const Shape& s, const void* x, const float* W, const float* bias, const float* tau,
                           const float* zp, const float* lse, void* o, bool reset, uint32_t* status, cudaStream_t st) {
  return SimtTiles<T>::deslice(s, in<T>(x), W, bias, tau, zp, lse, out<T>(o), reset, status, st);
}
template <typename T>
cudaError_t launch_bwd(const Shape& s, int mode, int P, const void* x, const void* dO, const void* fx,
                       const float* W, const float* bias, const float* tau, const float* zp, const float* dUS,
                       const float* lse, void* dx, void* dfx, float* delta, float* dt_part, float* part,
                       int accumulate, bool reset, uint32_t* status, cudaStream_t st) {
  return SimtTiles<T>::backward(s, mode, P, in<T>(x), in<T>(dO), in<T>(fx), W, bias, tau, zp, dUS, lse, out<T>(dx),
                                out<T>(dfx), delta, dt_part, part, accumulate, reset, status, st);
}

}  // namespace

cudaError_t simt_stats(const Shape& s, const void* x, const float* W, const float* bias, const float* tau,
                       float* lse, bool reset, uint32_t* status, cudaStream_t st) {
  return FS_DISPATCH(s, launch_stats, s, x, W, bias, tau, lse, reset, status, st);
}

cudaError_t simt_slice_partials(const Shape& s, int P, const void* x, const void* f, const float* W,
                                const float* bias, const float* tau, const float* lse, float* part,
                                bool reset, uint32_t* status, cudaStream_t st) {
  return FS_DISPATCH(s, launch_slice, s, P, x, f, W, bias, tau, lse, part, reset, status, st);
}

cudaError_t simt_reduce_tokens(const Shape& s, int P, const float* part, int Gs, float* tokens, float* wsum,
                               int finalize, cudaStream_t st) {
  const int64_t n = s.BH() * s.G * 32;  // a warp per output row
  return launch(k_reduce_tokens, dim3((unsigned)((n + 255) / 256)), dim3(256), 0, st, part, P, s.BH(), s.G, Gs, s.d,
                tokens, wsum, finalize, s.eps);
}

cudaError_t simt_finalize(const Shape& s, float* tokens, const float* wsum, cudaStream_t st) {
  const int64_t BHG = s.BH() * s.G;
  return launch(k_finalize, dim3((unsigned)((BHG * s.d + 255) / 256)), dim3(256), 0, st, tokens, wsum, BHG, s.d, s.eps);
}

cudaError_t simt_mix(const Shape& s, const float* M, const float* z, float* zp, cudaStream_t st) {
  const dim3 grid((unsigned)((s.G + kMixTG - 1) / kMixTG), (unsigned)s.BH(), (unsigned)((s.d + kMixTC - 1) / kMixTC));
  return launch(s.G % 4 == 0 ? k_mix_tiled<false, true> : k_mix_tiled<false, false>, grid, dim3(256), 0, st, M, z, zp,
                s.H, s.G, s.d);
}

cudaError_t simt_mix_bwd(const Shape& s, const float* M, const float* z, const float* dzp, float* dz, float* dM,
                         cudaStream_t st) {
  const dim3 grid((unsigned)((s.G + kMixTG - 1) / kMixTG), (unsigned)s.BH(), (unsigned)((s.d + kMixTC - 1) / kMixTC));
  cudaError_t e = launch(s.G % 4 == 0 ? k_mix_tiled<true, true> : k_mix_tiled<true, false>, grid, dim3(256), 0, st, M,
                         dzp, dz, s.H, s.G, s.d);
  if (e != cudaSuccess) return e;
  const dim3 tiles((unsigned)((s.G + 63) / 64), (unsigned)((s.G + 63) / 64), (unsigned)s.H);
  return launch(k_mix_bwd_dM, tiles, dim3(256), 0, st, z, dzp, dM, s.B, s.H, s.G, s.d);
}

cudaError_t simt_mix_channels(const Shape& s, const float* Wc, const float* z, float* zp, cudaStream_t st) {
  const int64_t BHG = s.BH() * s.G;
  return launch(k_mix_channels<false>, dim3((unsigned)((BHG * s.d + 255) / 256)), dim3(256), 0, st, Wc, z, zp, BHG, s.H,
                s.G, s.d);
}

cudaError_t simt_mix_channels_bwd(const Shape& s, const float* Wc, const float* z, const float* dzp, float* dz,
                                  float* dWc, cudaStream_t st) {
  const int64_t BHG = s.BH() * s.G;
  cudaError_t e = launch(k_mix_channels<true>, dim3((unsigned)((BHG * s.d + 255) / 256)), dim3(256), 0, st, Wc, dzp, dz,
                         BHG, s.H, s.G, s.d);
  if (e != cudaSuccess) return e;
  const int64_t n = (int64_t)s.H * s.d * s.d;
  return launch(k_mix_channels_dW, dim3((unsigned)((n + 127) / 128)), dim3(128), 0, st, z, dzp, dWc, s.B, s.H, s.G,
                s.d);
}

cudaError_t simt_deslice(const Shape& s, const void* x, const float* W, const float* bias, const float* tau,
                         const float* zp, const float* lse, void* o, bool reset, uint32_t* status, cudaStream_t st) {
  return FS_DISPATCH(s, launch_deslice, s, x, W, bias, tau, zp, lse, o, reset, status, st);
}

cudaError_t simt_deslice_bwd(const Shape& s, int P, const void* x, const float* W, const float* bias,
                             const float* tau, const float* zp, const float* lse, const void* dout, float* dzp,
                             void* dx, float* dW, float* db, float* dtau, int accumulate, float* delta,
                             float* part, float* dt_part, bool reset, uint32_t* status, cudaStream_t st) {
  cudaError_t e = FS_DISPATCH(s, launch_bwd, s, 0, P, x, dout, nullptr, W, bias, tau, zp, nullptr, lse, dx, nullptr,
                              delta, dt_part, part, accumulate, reset, status, st);
  if (e != cudaSuccess) return e;
  return simt_reduce_bwd(s, P, part, s.G, 2 * s.d + 2, 1, tau, dzp, dW, db, dtau, dt_part, simt_point_blocks(s),
                         accumulate, st);
}

cudaError_t simt_slice_bwd(const Shape& s, int P, const void* x, const void* f, const float* W,
                           const float* bias, const float* tau, const float* z, const float* wsum,
                           const float* lse, const float* dz, void* dx, void* dfx, float* dW, float* db,
                           float* dtau, int accumulate, float* delta, float* dUS, float* part, float* dt_part,
                           bool reset, uint32_t* status, cudaStream_t st) {
  cudaError_t e = simt_slice_bwd_prep(s, z, wsum, dz, dUS, st);
  if (e != cudaSuccess) return e;
  e = FS_DISPATCH(s, launch_bwd, s, 1, P, x, nullptr, f, W, bias, tau, nullptr, dUS, lse, dx, dfx, delta, dt_part,
                  part, accumulate, reset, status, st);
  if (e != cudaSuccess) return e;
  return simt_reduce_bwd(s, P, part, s.G, s.d + 2, 0, tau, nullptr, dW, db, dtau, dt_part, simt_point_blocks(s),
                         accumulate, st);
}

// The coupling's whole backward on the SIMT kernels: d z' as the forward slice's
// unnormalised numerators with dO for fx, the mix backward, the slice's dU, dS, then
// one point pass and one slot pass for da_D + da_S (mode 2)
// and the parameter reductions.  `part` holds the larger of the two partial sets;
// the d z' reduction's weight sums go to dUS, which the prologue then overwrites.
cudaError_t simt_coupling_bwd(const Shape& s, int P, const void* x, const void* fx, const void* dout,
                              const float* W, const float* bias, const float* tau, const float* M, const float* z,
                              const float* wsum, const float* zp, const float* lse, float* dzp, float* dz,
                              float* dM, void* dx, void* dfx, float* dW, float* db, float* dtau, int accumulate,
                              float* delta, float* dUS, float* part, float* dt_part, bool reset, uint32_t* status,
                              cudaStream_t st) {
  cudaError_t e = simt_slice_partials(s, P, x, dout, W, bias, tau, lse, part, reset, status, st);
  if (e != cudaSuccess) return e;
  if ((e = simt_reduce_tokens(s, P, part, s.G, dzp, dUS, 0, st)) != cudaSuccess) return e;
  if ((e = simt_mix_bwd(s, M, z, dzp, dz, dM, st)) != cudaSuccess) return e;
  if ((e = simt_slice_bwd_prep(s, z, wsum, dz, dUS, st)) != cudaSuccess) return e;
  e = FS_DISPATCH(s, launch_bwd, s, 2, P, x, dout, fx, W, bias, tau, zp, dUS, lse, dx, dfx, delta, dt_part, part,
                  accumulate, false, status, st);
  if (e != cudaSuccess) return e;
  return simt_reduce_bwd(s, P, part, s.G, s.d + 2, 0, tau, nullptr, dW, db, dtau, dt_part, simt_point_blocks(s),
                         accumulate, st);
}
// Kernels it launches (the statistics, when needed, are counted by the caller).
int simt_coupling_bwd_launch_count() { return 2 /*partials, reduce*/ + 2 /*mix backward*/ + 1 /*prologue*/ +
                                              2 /*point, slot*/ + 2 /*reductions*/; }

}  // namespace fs
