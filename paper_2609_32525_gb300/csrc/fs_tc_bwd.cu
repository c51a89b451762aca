// Tensor-core backward (tcgen05 / TMEM / TMA) for bf16 inputs on sm_103a.
//
// The gradients of the slice and of the deslice (Sec. 3.3) share one form.  With
// w_ng = softmax_g(a_ng), a per-point vector v_n and per-slot t_g, c_g:
//   dw_ng = v_n . t_g + c_g,   delta_n = sum_g w_ng dw_ng,   da_ng = w_ng (dw_ng - delta_n)
//   deslice: v = dO, t = z', c = 0;   slice: v = fx, t = dU = dz/(S+eps), c = dS = -dz.z/(S+eps)
// and then
//   dx_n = (1/tau) sum_g da_ng W[:,g],   dW[:,g] = (1/tau) sum_n da_ng x_n,
//   dbias_g = (1/tau) sum_n da_ng,       dtau = -(1/tau) sum_n sum_g da_ng (a_ng - lse_n),
//   deslice also d z'_g = sum_n w_ng dO_n;  slice also dfx_n = sum_g w_ng dU_g.
// Three passes, w recomputed in each and never written to memory:
//   rows  (point-owned; the deslice kernel in a backward mode): delta_n (and dfx_n);
//   slot  (slot-owned, split over points): dW, dbias, dtau (and d z') partials;
//   point (point-owned): dx.
// dw - delta is one more MMA chain of the logits' shape: the slot side carries
// [t_g | c_g halves, 1, 1, 1] (the T image, laid out as the W image) and the point
// side [v_n | 1, 1, -delta_n in three bf16 parts] (delta's point-extra rows).
#include "fs_tc_common.cuh"

namespace fs {
namespace {

using namespace tc;

constexpr int kBStages = 6;                            // slot pass pipeline depth (point tiles)
constexpr int kDxStages = 3;                           // point pass pipeline depth
constexpr uint32_t kBStage = 2 * kXBytes + 2 * kPxBytes;  // x | v | lse rows | delta rows (TMA halves)
constexpr uint32_t kPxZero = 2 * kPxBytes;             // one zero block for the k = 8..15 halves
constexpr uint32_t kWBlockB = kGC * kWRow;             // one 128-slot block of a W or T image

// ---- prep kernels ------------------------------------------------------------------------------

// The slice's token gradients as images: per (b,h) and slot, u_g = dz_g / (S_g + eps) and
// c_g = -(dz_g . z_g) / (S_g + eps).  T image in the W image's layout (kWRow bytes per slot):
// u rounded to bf16, the extra rows [c_hi, c_lo, 1, 1, 1, 0...] (k = 2..4 meet -delta's three
// parts), the residuals; the Z-layout image of u (hi, then residual); c itself.  Padding
// slots [G, Gp) get u = 0 and c = 0 (their weights are 0).
// A block takes 64 slots of one (b,h): a warp per slot row, then 16-byte pieces of the images
// from shared memory.
__global__ void __launch_bounds__(256) k_prep_us(const float* __restrict__ z, const float* __restrict__ wsum,
                                                 const float* __restrict__ dz, uint8_t* __restrict__ timg,
                                                 uint8_t* __restrict__ zimg, float* __restrict__ c_out, int G, int Gp,
                                                 float eps) {
  grid_begin(z, wsum, dz);
  __shared__ float su[64][kD + 1];
  const int64_t bh = blockIdx.y;
  const int g0 = blockIdx.x * 64, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  uint8_t* base = timg + (size_t)bh * Gp * kWRow;
#pragma unroll
  for (int i = 0; i < 8; i++) {
    const int w = warp * 8 + i, g = g0 + w;
    const bool real = g < G;
    const int64_t row = (bh * G + (real ? g : 0)) * kD + lane;
    const float d = real ? dz[row] : 0.f;
    const float den = real ? wsum[bh * G + g] + eps : 1.f;
    float s = real ? d * z[row] : 0.f;
#pragma unroll
    for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    su[w][lane] = d / den;
    if (lane == 0) {
      const float c = -s / den;
      c_out[bh * Gp + g] = c;
      const uint32_t hi = pack_bf16(c, 0.f) & 0xFFFFu;
      const uint32_t lo = pack_bf16(c - __uint_as_float(hi << 16), 0.f) & 0xFFFFu;
      uint8_t* ep = base + (size_t)Gp * 64;
      *reinterpret_cast<uint4*>(ep + off_sw32(g, 0)) = make_uint4(hi | (lo << 16), 0x3F803F80u, 0x3F80u, 0u);
      *reinterpret_cast<uint4*>(ep + off_sw32(g, 8)) = make_uint4(0u, 0u, 0u, 0u);
    }
  }
  __syncthreads();
  {
    const int w = threadIdx.x >> 2, q = threadIdx.x & 3;
    float v[8];
#pragma unroll
    for (int e = 0; e < 8; e++) v[e] = su[w][8 * q + e];
    const uint32_t off = off_sw64(g0 + w, 8 * q);
    split8(v, *reinterpret_cast<uint4*>(base + off), *reinterpret_cast<uint4*>(base + (size_t)Gp * 96 + off));
  }
  {
    const int c = threadIdx.x & 31, w8 = threadIdx.x >> 5;
    float v[8];
#pragma unroll
    for (int e = 0; e < 8; e++) v[e] = su[w8 * 8 + e][c];
    uint8_t* zi = zimg + (size_t)bh * Gp * 128 + off_z(c, g0 + w8 * 8);
    split8(v, *reinterpret_cast<uint4*>(zi), *reinterpret_cast<uint4*>(zi + (size_t)Gp * 64));
  }
}

// delta's point-extra rows [1, 1, -delta in three bf16 parts, 0, 0, 0] into dpx [BH, Np, 8];
// delta_n = delta[bh][n] (+ delta2[bh][n] when given, + the nwds (two or three) partials
// wds[.][bh][n] when wds is given).
__global__ void k_prep_dpx(const float* __restrict__ delta, const float* __restrict__ delta2,
                           const float* __restrict__ wds, int nwds, uint4* __restrict__ dpx, int64_t BH, int64_t N,
                           int64_t Np) {
  grid_begin(delta, delta2, wds);
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= BH * Np) return;
  const int64_t bh = i / Np, n = i % Np;
  float d = 0.f;
  if (n < N) {
    d = delta[bh * N + n];
    if (delta2) d += delta2[bh * N + n];
    if (wds) {
      float w = wds[bh * N + n] + wds[(BH + bh) * N + n];
      if (nwds == 3) w += wds[(2 * BH + bh) * N + n];
      d += w;
    }
  }
  dpx[i] = extra_row3(-d);
}

// ---- device pieces -----------------------------------------------------------------------------

// M = 128 x N = 64 product with K = 48 (80 with the residual half, lo of A or B): a, b the
// low descriptor words of the K-major 64B-swizzled 32-channel blocks, ae, be those of the
// extra blocks with high words kAeHi, kBeHi (kAeHi = 0: K = 32 / 64, no extra block).
// acc0: add to what d holds (a second chain into the same accumulator).
template <bool kLoA, uint32_t kAeHi, uint32_t kBeHi>
__device__ __forceinline__ void issue_dot64(uint32_t d, uint32_t a, uint32_t b, uint32_t ae, uint32_t be, uint32_t lo,
                                            uint32_t acc0 = 0) {
  constexpr uint32_t idesc = idesc_bf16(128, 64, false, false);
  mma_ss_w<kHi64, kHi64>(d, a, b, idesc, acc0);
  mma_ss_w<kHi64, kHi64>(d, a + 2, b + 2, idesc, 1);
  if (lo) {
    mma_ss_w<kHi64, kHi64>(d, kLoA ? lo : a, kLoA ? b : lo, idesc, 1);
    mma_ss_w<kHi64, kHi64>(d, kLoA ? lo + 2 : a + 2, kLoA ? b + 2 : lo + 2, idesc, 1);
  }
  if (kAeHi != 0) mma_ss_w<kAeHi, kBeHi>(d, ae, be, idesc, 1);
}

// The main part of the same product with the slot side (A) in TMEM: tA holds a slot
// block's rows as packed bf16 pairs, K steps of 8 columns: the bf16 half (2 steps), its
// residual (2).  Only the point side (B) is read from shared memory.
__device__ __forceinline__ void issue_dot64_ts(uint32_t d, uint32_t tA, uint32_t b, bool lo) {
  constexpr uint32_t idesc = idesc_bf16(128, 64, false, false);
  mma_ts_w<kHi64>(d, tA, b, idesc, 0u);
  mma_ts_w<kHi64>(d, tA + 8, b + 2, idesc, 1u);
  if (lo) {
    mma_ts_w<kHi64>(d, tA + 16, b, idesc, 1u);
    mma_ts_w<kHi64>(d, tA + 24, b + 2, idesc, 1u);
  }
}

// Low word of a point-extra descriptor (no swizzle, 16-byte rows) whose k = 8..15 half is
// the shared zero block; n rows further on both its fields change.
__device__ __forceinline__ uint32_t px_lo(uint32_t px_s, uint32_t zero_s) { return sdesc_lo(px_s, zero_s - px_s); }

// One half (32 columns) of a unit of a TMEM lane: L (log2 weights) at tL, dw - delta at tD.
// da = 2^L (dw - delta) goes back in place into the L columns as bf16 pairs: columns
// [0, 16) the hi halves of the 32 entries, [16, 32) their lo halves (kSplit).  kW: the
// weights too, into the dw columns, same layout.
// kSums: dt += sum da L, db += sum da.
// loaded(): called once the half's columns are in registers.
template <bool kSplit, bool kW, bool kSums, typename F>
__device__ __forceinline__ void da_half(uint32_t tL, uint32_t tD, float& dt, float& db, F loaded) {
  // Pairs of entries go through the packed f32x2 forms (one instruction for both).
  const uint64_t neg1 = pack2(__float_as_uint(-1.f), __float_as_uint(-1.f));
  uint32_t l[32], dw[32];
  tmem_ld32(tL, l);
  tmem_ld32(tD, dw);
  tmem_wait_ld2(l, dw);
  loaded();
  uint32_t dh[16], dl[16], wh[16], wl[16];
  uint64_t t2 = 0, sb2 = 0;  // (+0, +0)
#pragma unroll
  for (int k = 0; k < 16; k++) {
    const uint64_t L2 = pack2(l[2 * k], l[2 * k + 1]);
    const uint64_t w2 = pack2(__float_as_uint(ex2(__uint_as_float(l[2 * k]))),
                              __float_as_uint(ex2(__uint_as_float(l[2 * k + 1]))));
    const uint64_t a2 = mul2(w2, pack2(dw[2 * k], dw[2 * k + 1]));
    if (kSums) {
      t2 = fma2(a2, L2, t2);
      sb2 = add2(sb2, a2);
    }
    const uint32_t p = pack_bf16(lo_f(a2), hi_f(a2));
    dh[k] = p;
    if (kSplit) {
      const uint64_t r2 = fma2(pack2(p << 16, p & 0xFFFF0000u), neg1, a2);  // a - bf16(a)
      dl[k] = pack_bf16(lo_f(r2), hi_f(r2));
    }
    if (kW) {
      const uint32_t q = pack_bf16(lo_f(w2), hi_f(w2));
      wh[k] = q;
      if (kSplit) {
        const uint64_t r2 = fma2(pack2(q << 16, q & 0xFFFF0000u), neg1, w2);
        wl[k] = pack_bf16(lo_f(r2), hi_f(r2));
      }
    }
  }
  tmem_st16(tL, dh);
  if (kSplit) tmem_st16(tL + 16, dl);
  if (kW) {
    tmem_st16(tD, wh);
    if (kSplit) tmem_st16(tD + 16, wl);
  }
  if (kSums) {
    dt += lo_f(t2) + hi_f(t2);
    db += lo_f(sb2) + hi_f(sb2);
  }
}

// One half of a unit: L (log2 weights) -> w = 2^L in place, as bf16 pairs in da_half's
// layout (hi pairs, then their residuals with kSplit).
template <bool kSplit>
__device__ __forceinline__ void w_half(uint32_t tL) {
  const uint64_t neg1 = pack2(__float_as_uint(-1.f), __float_as_uint(-1.f));
  uint32_t l[32];
  tmem_ld32(tL, l);
  tmem_wait_ld(l);
  uint32_t wh[16], wl[16];
#pragma unroll
  for (int k = 0; k < 16; k++) {
    const uint64_t w2 = pack2(__float_as_uint(ex2(__uint_as_float(l[2 * k]))),
                              __float_as_uint(ex2(__uint_as_float(l[2 * k + 1]))));
    const uint32_t q = pack_bf16(lo_f(w2), hi_f(w2));
    wh[k] = q;
    if (kSplit) {
      const uint64_t r2 = fma2(pack2(q << 16, q & 0xFFFF0000u), neg1, w2);
      wl[k] = pack_bf16(lo_f(r2), hi_f(r2));
    }
  }
  tmem_st16(tL, wh);
  if (kSplit) tmem_st16(tL + 16, wl);
}

// TMEM buffers of a unit's logits L (which become da) and of its dw - delta.  da stays until
// its products have read it; dw - delta is dead once a softmax warp has loaded it, so two
// buffers of it feed four of L and four units are under way instead of three.  (The slot
// pass's MODE 1 writes the weights over dw, for its second product: three of each.)
template <bool kKeepDw>
struct UnitBufs {
  static constexpr int kL = kKeepDw ? 3 : 4, kD = kKeepDw ? 3 : 2;
  static constexpr uint32_t kDCol = kL * 64;  // column of the first dw buffer
};

// The slot pass's accumulators are flushed into registers every kSlotFlush of an
// issuer's units (64 points each), for the reason the slice's are: the tensor cores'
// fp32 accumulation drifts towards zero over a long chain of K steps.
constexpr int kSlotFlush = 8;
__device__ __forceinline__ bool slot_flush_at(int u) { return ((u >> 1) % kSlotFlush) == 0; }

// =========================================================================================
// Slot pass: CTA (slot block, point split p, bh) owns 128 slots.  Unit u is half
// u & 1 (64 points) of point tile u >> 1.  Per unit, warp 1 forms, transposed
// (M = 128 slots, N = 64 points, TMEM lane = slot),
//   L = a2 - lse2 (W block vs [x | 1, 1, -lse2]) and dw - delta (T block vs [v | 1, 1, -delta]);
// (warp 2 the latter); softmax warpgroup u % 2 turns them into da (and, MODE 1, w) in place,
// a half at a time, and sums da (a2 - lse2) and da per slot in registers; warp 3 issues, per half,
//   dWx += da^T x   (K = points; x's 64B-swizzled tile read as an MN-major B operand)
//   MODE 1: dZ += w^T dO (the token gradient), from dO's tile the same way.
// Writes part[p][bh][g] = MODE 1: (dZ(32), dWx(32), sum da, 0); MODE 2: (dWx, sum da, 0)
// and dt_part[bh][p * R + block] = ln2 * sum over the block's slots of sum da (a2 - lse2).
// Two more modes serve fs_coupling_bwd:
//   MODE 0: the token gradient alone, dZ += w^T dO (no dw chain, no da): part = dZ(32);
//   MODE 3: da = da_D + da_S as in the combined point pass (dw - delta as two chains:
//     the deslice's T block against dO, the slice's T2 block against [fx | 1, 1, -delta]
//     (its extra block [dS_hi, dS_lo, 1, 1, 1] meets delta's rows), delta = delta_D +
//     delta_S), written like MODE 2.
// smem: [W block: hi 8K | extra 4K | lo 8K][T block: same][stages][zero 2K][red 1.5K][bars]
// TMEM: [0, 384) the units' L and dw buffers (UnitBufs); accumulators dWx_j [384 + 32 j),
// dZ_j [448 + 32 j).
//
// What bounds it is the cycle of a unit's buffers (logits -> da -> products -> logits): ~1100
// clocks a unit where the MMAs alone need ~750 and the exponentials 256; the softmax warps wait
// half of their time.  So the halves of a unit are handed over as they are written, and four
// units are under way.  Whole backward at B = 2, N = 131,072, H = 8, G = 512, this pass and the
// point pass changed together: 2261 us with whole units, two warps issuing the products and
// three units under way; 2198 with halves (and the point pass's third warpgroup), 2184 with one
// warp per chain, 2165 with four units.
// =========================================================================================
template <int MODE, bool split>
__global__ void __launch_bounds__(kThreads, 1)
    k_bwd_slot_tc(const __grid_constant__ CUtensorMap xmap, const __grid_constant__ CUtensorMap vmap,
                  const __grid_constant__ CUtensorMap pmap, const __grid_constant__ CUtensorMap dmap,
                  const __grid_constant__ CUtensorMap fmap, const uint8_t* __restrict__ wimg,
                  const uint8_t* __restrict__ timg, const uint8_t* __restrict__ timg2, float* __restrict__ part,
                  float* __restrict__ dt_part, int64_t N, int64_t Np, int H, int G, int splits,
                  uint32_t* status) {
  constexpr int kNSt = MODE == 3 ? kBStages - 1 : kBStages;    // stages (MODE 3's are larger)
  constexpr uint32_t kStgS = kBStage + (MODE == 3 ? kXBytes : 0u);  // x | v | px | dpx [| fx]
  const int g_base = blockIdx.x * kGC;
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* s_w = smem;               // W block
  uint8_t* s_t = s_w + kWBlockB;     // T block
  uint8_t* s_t2 = s_t + kWBlockB;    // MODE 3: the slice's T block
  uint8_t* s_st = s_t2 + (MODE == 3 ? kWBlockB : 0u);  // stages
  uint8_t* s_zero = s_st + kNSt * kStgS;  // above the stages' point rows (positive LBO)
  float* s_red = reinterpret_cast<float*>(s_zero + kPxZero);  // 3 x 128 floats
  uint64_t* bars = reinterpret_cast<uint64_t*>(s_red + 3 * kGC);
  uint64_t* w_full = bars;
  uint64_t* x_full = bars + 1;
  uint64_t* st_empty = x_full + kNSt;
  uint64_t* s_full = st_empty + kNSt;
  using Bufs = UnitBufs<MODE == 1>;
  uint64_t* p_ready = s_full + Bufs::kL;  // [L buffer][half of the unit]
  uint64_t* pv_done = p_ready + 2 * Bufs::kL;
  uint64_t* dw_free = pv_done + Bufs::kL;
  uint64_t* acc_full = dw_free + Bufs::kD;
  uint64_t* acc_done = acc_full + 1;  // [half][its units' parity]: a unit's products complete
  uint64_t* wt_ready = acc_done + 4;  // MODES 2, 3: the W' image is in TMEM
  uint64_t* drain = wt_ready + 1;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain + 3);
  Abort* ab = reinterpret_cast<Abort*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const Work wk = work_of(N, splits, blockIdx.y, blockIdx.z);
  const int64_t b = wk.bh / H;
  const int h = (int)(wk.bh % H);
  const int units = 2 * wk.ntiles;
  // Accumulator flushes (as in the slice): issuer j's chain restarts every
  // kSlotFlush of its units after warpgroup j has added the accumulator into
  // registers.  MODE 1 keeps two accumulators per issuer (dW, dZ) and no flushes.
  constexpr bool kFl = MODE != 1;
  // MODES 2 and 3 keep no dZ accumulator, so its 64 TMEM columns hold slot-side images
  // and those MMAs read only their point side from shared memory: MODE 2 the W' image
  // (W', its residual, the extra block: 40 columns); MODE 3 W' and its residual (32)
  // and the deslice's T image and its residual (32), the two extra blocks staying in
  // shared memory.
  constexpr bool kWT = MODE == 2 || MODE == 3;
  constexpr bool kTT = MODE == 3;
  constexpr uint32_t kAccW = 384u, kAccZ = kAccW + 64;
  constexpr uint32_t kAccF = MODE == 0 ? kAccZ : kAccW;  // the flushed accumulator
  constexpr uint32_t kVOff = kXBytes, kPOff = 2 * kXBytes, kDOff = 2 * kXBytes + kPxBytes;

  if (threadIdx.x == 0) {
    mbar_init(w_full, 1);
    for (int s = 0; s < kNSt; s++) {
      mbar_init(&x_full[s], 1);
      mbar_init(&st_empty[s], MODE == 0 ? 2 : 3);  // the issuers
    }
    for (int i = 0; i < Bufs::kL; i++) {
      mbar_init(&s_full[i], MODE == 0 ? 1 : 2);  // logits and dw
      mbar_init(&p_ready[2 * i], 4);
      mbar_init(&p_ready[2 * i + 1], 4);
      mbar_init(&pv_done[i], 1);
    }
    for (int i = 0; i < Bufs::kD; i++) mbar_init(&dw_free[i], 4);
    mbar_init(acc_full, 1);
    for (int i = 0; i < 4; i++) mbar_init(&acc_done[i], 1);
    mbar_init(wt_ready, 4);
    for (int i = 0; i < 3; i++) mbar_init(&drain[i], 1);
    ab->flag = 0;
    fence_mbar_init();
  }
  zero_smem(s_zero, kPxZero);
  fence_proxy_async_smem();
  if (warp == 1) tmem_alloc(tmem_slot, 512);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  grid_trigger();
  grid_wait(wimg, timg, timg2);

  if (warp == 0) {
    // ------------------------------ producer ------------------------------
    if (lane == 0) {
      prefetch_tmap(&xmap);
      prefetch_tmap(&vmap);
      prefetch_tmap(&pmap);
      if (MODE != 0) prefetch_tmap(&dmap);
      if (MODE == 3) prefetch_tmap(&fmap);
      constexpr int kImages = MODE == 0 ? 1 : (MODE == 3 ? 3 : 2);  // W [, T [, T2]]
      mbar_expect_tx(w_full, kImages * kWBlockB);
      const uint8_t* ws = wimg + (size_t)h * G * kWRow;
      const uint8_t* ts = timg + (size_t)wk.bh * G * kWRow;
      const uint8_t* ts2 = MODE == 3 ? timg2 + (size_t)wk.bh * G * kWRow : nullptr;
      for (int im = 0; im < kImages; im++) {
        const uint8_t* src = im == 0 ? ws : (im == 1 ? ts : ts2);
        uint8_t* dst = im == 0 ? s_w : (im == 1 ? s_t : s_t2);
        load_images(dst, src + (size_t)g_base * 64, kGC * 64, w_full);
        load_images(dst + kGC * 64, src + (size_t)G * 64 + (size_t)g_base * 32, kGC * 32, w_full);
        load_images(dst + kGC * 96, src + (size_t)G * 96 + (size_t)g_base * 64, kGC * 64, w_full);
      }
      int i = 0;
      for (; i < wk.ntiles; i++) {
        const int s = i % kNSt;
        if (i >= kNSt && !mbar_wait(&st_empty[s], (uint32_t)(((i / kNSt) - 1) & 1), ab, status)) break;
        uint8_t* st = s_st + s * kStgS;
        const int n0 = (int)((wk.tile0 + i) * kTile);
        mbar_expect_tx(&x_full[s], MODE == 0 ? kBStage - kPxBytes : kStgS);
        tma_load_3d(st, &xmap, h * kD, n0, (int)b, &x_full[s]);
        tma_load_3d(st + kVOff, &vmap, h * kD, n0, (int)b, &x_full[s]);
        tma_load_2d(st + kPOff, &pmap, 0, (int)(wk.bh * Np + n0), &x_full[s]);
        if (MODE != 0) tma_load_2d(st + kDOff, &dmap, 0, (int)(wk.bh * Np + n0), &x_full[s]);
        if (MODE == 3) tma_load_3d(st + kBStage, &fmap, h * kD, n0, (int)b, &x_full[s]);
      }
      for (int j = (i > kNSt ? i - kNSt : 0); j < i; j++)
        mbar_wait(&x_full[j % kNSt], (uint32_t)((j / kNSt) & 1), ab, nullptr, kWaitNs);
      mbar_wait(w_full, 0, ab, nullptr, kWaitNs);
    }
  } else if (warp == 1 || (warp == 2 && MODE != 0)) {
    // ------------------------------ logits (warp 1) and dw (warp 2) issuers ------------------------------
    const uint32_t w = sdesc_lo(smem_u32(s_w), 16), t = sdesc_lo(smem_u32(s_t), 16), t2 = sdesc_lo(smem_u32(s_t2), 16);
    const uint32_t sz = smem_u32(s_zero);
    constexpr uint32_t kExt = kGC * 4, kLo = kGC * 6;  // the extra and residual rows of a slot block, in 16 bytes
    bool ok = mbar_wait_w(w_full, 0, ab, status);
    if (kWT && ok) {
      ok = mbar_wait_w(wt_ready, 0, ab, status);
      tc_fence_after();
    }
    Ring<kNSt> stg;
    Ring<Bufs::kL> sb;
    Ring<Bufs::kD> db;
    for (int i = 0, u = 0; ok && i < wk.ntiles; i++, stg.next()) {
      if (!(ok = mbar_wait_w(&x_full[stg.i], stg.pass, ab, status))) break;
      const uint32_t st = smem_u32(s_st + stg.i * kStgS);
      uint32_t x = sdesc_lo(st, 16);
      uint32_t px = px_lo(st + (warp == 1 ? kPOff : kDOff), sz);  // lse's rows, delta's rows
      // the second half's 64 points: 64-byte-row tiles, then 16-byte extra rows (whose
      // leading offset to the zero block shrinks as the address grows)
      constexpr uint32_t kHalf = 64 * 64 / 16, kHalfP = 64 * 16 / 16 - ((64u * 16 / 16) << 16);
#pragma unroll 1
      for (int half = 0; half < 2; half++, u++, sb.next(), db.next(), x += kHalf, px += kHalfP) {
        // L: the products of the unit kL back; dw: loaded by the unit kD back
        const bool is_l = warp == 1 || MODE == 1;
        if (u >= (is_l ? Bufs::kL : Bufs::kD) &&
            !(ok = mbar_wait_w(is_l ? &pv_done[sb.i] : &dw_free[db.i], (is_l ? sb.pass : db.pass) ^ 1u, ab, status)))
          break;
        tc_fence_after();
        const uint32_t tL = tmem + (uint32_t)sb.i * 64, tD = tmem + Bufs::kDCol + (uint32_t)db.i * 64;
        if (warp == 1) {
          if (kTT) {
            issue_dot64_ts(tL, tmem + kAccZ, x, split);
            mma_ss_w<kHi32, kHiPx>(tL, w + kExt, px, idesc_bf16(128, 64, false, false), 1u);
          } else if (kWT) {
            issue_dot64_ts(tL, tmem + kAccZ, x, split);
            mma_ts_w<kHiPx>(tL, tmem + kAccZ + 32, px, idesc_bf16(128, 64, false, false), 1u);
          } else {
            issue_dot64<true, kHi32, kHiPx>(tL, w, x, w + kExt, px, split ? w + kLo : 0u);
          }
        } else if (kTT) {
          // the deslice's chain: T (and its residual) from TMEM against dO, no extra block;
          // the slice's extra block [dS_hi, dS_lo, 1, 1, 1] against delta's rows
          // [1, 1, -delta parts] adds dS - delta in one K step.
          issue_dot64_ts(tD, tmem + kAccZ + 32, x + kVOff / 16, split);
          issue_dot64<true, kHi32, kHiPx>(tD, t2, x + kBStage / 16, t2 + kExt, px, split ? t2 + kLo : 0u, 1u);
        } else {
          issue_dot64<true, kHi32, kHiPx>(tD, t, x + kVOff / 16, t + kExt, px, split ? t + kLo : 0u);
        }
        mma_commit_w(&s_full[sb.i]);
      }
      mma_commit_w(&st_empty[stg.i]);
    }
    mma_commit_w(&drain[warp - 1]);
    mbar_wait_w(&drain[warp - 1], 0, ab, nullptr, kWaitNs);
  } else if (warp == 3) {
    // ------------------------------ product issuer ------------------------------
    // Units u (half u & 1 of every tile) into accumulator u & 1.
    constexpr uint32_t idesc = idesc_bf16(128, kD, false, true);
    bool ok = true;
    Ring<kNSt> stg;
    Ring<Bufs::kL> sb;
    Ring<Bufs::kD> db;
    for (int u = 0; ok && u < units; u++, sb.next(), db.next()) {
      const int j = u & 1;
      // 16 points: two 8-row groups of the 64B-swizzled tile (MN-major: channels contiguous).
      const uint32_t x = sdesc_lo(smem_u32(s_st + stg.i * kStgS) + (uint32_t)j * 64 * 64, 4096), v = x + kVOff / 16;
      const uint32_t tL = tmem + (uint32_t)sb.i * 64, tD = tmem + Bufs::kDCol + (uint32_t)db.i * 64;
      const uint32_t tW = tmem + kAccW + (uint32_t)j * 32, tZ = tmem + kAccZ + (uint32_t)j * 32;
      const bool fresh = u < 2 || (kFl && slot_flush_at(u));
#pragma unroll
      for (int kk = 0; kk < 4; kk++) {
        if ((kk & 1) == 0) {  // a half of the unit
          if (!(ok = mbar_wait_w(&p_ready[2 * sb.i + (kk >> 1)], sb.pass, ab, status))) break;
          tc_fence_after();
        }
        const uint32_t acc = (!fresh || kk > 0) ? 1u : 0u;
        if (MODE == 0) {  // the weights are in the L columns: dZ += w^T dO
          mma_ts_w<kHi64>(tZ, tL + da_col(kk), v + kk * 64, idesc, acc);
          if (split) mma_ts_w<kHi64>(tZ, tL + da_col(kk) + 16, v + kk * 64, idesc, 1u);
          continue;
        }
        mma_ts_w<kHi64>(tW, tL + da_col(kk), x + kk * 64, idesc, acc);
        if (split) mma_ts_w<kHi64>(tW, tL + da_col(kk) + 16, x + kk * 64, idesc, 1u);
        if (MODE == 1) {
          mma_ts_w<kHi64>(tZ, tD + da_col(kk), v + kk * 64, idesc, acc);
          if (split) mma_ts_w<kHi64>(tZ, tD + da_col(kk) + 16, v + kk * 64, idesc, 1u);
        }
      }
      mma_commit_w(&pv_done[sb.i]);
      if (kFl) mma_commit_w(&acc_done[acc_done_of(u)]);
      if (j == 1) {
        mma_commit_w(&st_empty[stg.i]);
        stg.next();
      }
    }
    if (ok) mma_commit_w(acc_full);
    mma_commit_w(&drain[2]);
    mbar_wait_w(&drain[2], 0, ab, nullptr, kWaitNs);
  } else if (warp >= kSoftmaxWarp0) {
    // ------------------------------ softmax warpgroups ------------------------------
    const int wg = (warp - kSoftmaxWarp0) >> 2;
    const int wq = warp & 3;
    const int r = wq * 32 + lane;  // TMEM lane: slot g_base + r
    const uint32_t lane_addr = (uint32_t)(wq * 32) << 16;
    bool ok = true;
    float dt = 0.f, db = 0.f;
    if (kWT && wg == 0) {
      // Slot r's W' row from the block's image in shared memory (64B / 32B swizzled
      // rows) into TMEM columns [kAccZ, kAccZ + 48) of lane r: packed bf16 pairs of W'
      // (16), its residual (16), the extra block (8, then 8 zero columns).
      if ((ok = mbar_wait(w_full, 0, ab, status))) {
        const uint32_t tW = tmem + lane_addr + kAccZ;
        // a slot-block image's row r: bf16 pairs of the main half and of the residual
        auto copy_rows = [&](const uint8_t* img, uint32_t tdst) {
          uint32_t hi[16], lo[16];
#pragma unroll
          for (int c = 0; c < 16; c++) {
            hi[c] = *reinterpret_cast<const uint32_t*>(img + off_sw64(r, 2 * c));
            lo[c] = split ? *reinterpret_cast<const uint32_t*>(img + kGC * 96 + off_sw64(r, 2 * c)) : 0u;
          }
          tmem_st16(tdst, hi);
          tmem_st16(tdst + 16, lo);
        };
        copy_rows(s_w, tW);
        if (kTT) {
          copy_rows(s_t, tW + 32);
        } else {
          uint32_t ex[16];
#pragma unroll
          for (int c = 0; c < 16; c++)
            ex[c] = c < 8 ? *reinterpret_cast<const uint32_t*>(s_w + kGC * 64 + off_sw32(r, 2 * c)) : 0u;
          tmem_st16(tW + 32, ex);
        }
        tmem_wait_st();
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(wt_ready);
    }
    float acc[kD];  // this warpgroup's flushed share of dWx (MODE 0: dZ)
#pragma unroll
    for (int k = 0; k < kD; k++) acc[k] = 0.f;
    auto add_acc = [&]() {
      uint32_t a[32];
      tmem_ld32(tmem + lane_addr + kAccF + (uint32_t)wg * 32, a);
      tmem_wait_ld(a);
#pragma unroll
      for (int k = 0; k < kD; k++) acc[k] += __uint_as_float(a[k]);
    };
    for (int u = wg; ok && u < units; u += 2) {
      const int bb = u % Bufs::kL, bd = u % Bufs::kD;
      if (!(ok = mbar_wait(&s_full[bb], (uint32_t)((u / Bufs::kL) & 1), ab, status))) break;
      tc_fence_after();
      const uint32_t tL = tmem + lane_addr + (uint32_t)bb * 64;
      const uint32_t tD = tmem + lane_addr + Bufs::kDCol + (uint32_t)bd * 64;
#pragma unroll
      for (int hf = 0; hf < 2; hf++) {
        if constexpr (MODE == 0) {
          w_half<split>(tL + 32 * hf);
        } else {
          da_half<split, MODE == 1, true>(tL + 32 * hf, tD + 32 * hf, dt, db, [&]() {
            if (MODE != 1 && hf == 1) {
              tc_fence_before();
              __syncwarp();
              if (lane == 0) mbar_arrive(&dw_free[bd]);
            }
          });
        }
        tmem_wait_st();
        if (hf == 0 && kFl && u >= 2 && slot_flush_at(u)) {
          // This warpgroup's units up to u - 2 have completed their products.
          if (!(ok = mbar_wait(&acc_done[acc_done_of(u - 2)], acc_done_phase(u - 2), ab, status))) break;
          tc_fence_after();
          add_acc();
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&p_ready[2 * bb + hf]);
      }
    }
    // Epilogue.  The block's partial rows are gathered in the stages' memory (every load has
    // landed and been read) and leave as one bulk copy.  Warpgroup 1 hands its sums dt, db to
    // warpgroup 0 the same way.  Flushed modes: each warpgroup adds what its accumulator holds
    // since its last flush, and the two shares are added in a fixed order (MODE 0: dZ; MODES 2,
    // 3: dWx and the sums).  MODE 1: warpgroup 0 writes dWx (both accumulators) and the sums,
    // warpgroup 1 dZ.
    const int64_t BH = gridDim.z;
    constexpr int PS = MODE == 1 ? 2 * kD + 2 : (MODE == 0 ? kD : kD + 2);
    float* s_out = reinterpret_cast<float*>(s_st);
    float* o = s_out + r * PS;
    const bool have = ok && wk.ntiles > 0 && mbar_wait(acc_full, 0, ab, status);
    if (have) tc_fence_after();
    if (kFl) {
      if (have) add_acc();
    } else if (have) {  // MODE 1: the sum of a product's two accumulators
      uint32_t a0[32], a1[32];
      tmem_ld32(tmem + lane_addr + (wg == 0 ? kAccW : kAccZ), a0);
      tmem_ld32(tmem + lane_addr + (wg == 0 ? kAccW : kAccZ) + 32, a1);
      tmem_wait_ld2(a0, a1);
#pragma unroll
      for (int k = 0; k < kD; k++) acc[k] = __uint_as_float(a0[k]) + __uint_as_float(a1[k]);
    }
    if (wg == 1) {
#pragma unroll
      for (int k = 0; k < kD; k++) o[k] = acc[k];
      if (MODE != 0) {
        s_red[r] = dt;
        s_red[kGC + r] = db;
      }
      fence_proxy_async_smem();
    }
    named_barrier(1, 256);
    if (wg == 0) {
#pragma unroll
      for (int k = 0; k < kD; k++) {
        if (kFl)
          o[k] = acc[k] + o[k];
        else
          o[kD + k] = acc[k];
      }
      if (MODE != 0) {
        dt += s_red[r];
        db += s_red[kGC + r];
        o[PS - 2] = db;
        o[PS - 1] = 0.f;
#pragma unroll
        for (int e = 16; e; e >>= 1) dt += __shfl_xor_sync(0xffffffffu, dt, e);
        if (lane == 0) s_red[2 * kGC + wq] = dt;
      }
      fence_proxy_async_smem();
      named_barrier(2, 128);
      if (r == 0) {
        if (MODE != 0)
          dt_part[wk.bh * ((int64_t)gridDim.x * gridDim.y) + (int64_t)blockIdx.y * gridDim.x + blockIdx.x] =
              ((s_red[2 * kGC] + s_red[2 * kGC + 1]) + (s_red[2 * kGC + 2] + s_red[2 * kGC + 3])) * kLn2;
        bulk_store(part + (((int64_t)blockIdx.y * BH + wk.bh) * G + g_base) * PS, s_out, kGC * PS * 4);
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 1) tmem_dealloc(tmem, 512);
}

// =========================================================================================
// Point pass: dx_n = ln2 * sum_g da_ng W'_g (W' = W log2(e)/tau) over slots [g0, g0 + G) of
// images of Gi slots; accumulate: added to what dx holds.  CTA (split, bh)
// walks its point tiles; block q is (tile q / nb, 64-slot chunk q % nb).  Warp 1
// forms L (x tile vs W rows) and warp 2 dw - delta (v tile vs T rows), M = 128 points,
// N = 64 slots; softmax warpgroup q % 3 writes da in place (hi, lo pairs), a half of the
// chunk at a time; warp 3 issues K-steps [2 j, 2 j + 2) of half j into O_j:
//   O_j += da W'^T (B: the W'^T image, channel rows, slots along K).
// kComb (the whole coupling's backward): da is the sum of the deslice's and the
// slice's, which share the weights, so one pass serves both: dw - delta is two chains
// into the same accumulator, dO against the deslice's T image (c = 0, so no extra
// block) and [fx | 1, 1, -delta] against the slice's (t = dU, c = dS): one extra K
// step adds dS - delta, with delta = delta_D + delta_S in the point rows.  Each stage
// also holds the fx tile.
// smem: [W img G x (96 | 160)][T img G x 96][kComb: T2 img G x 96][W'^T img G x 64]
//       [stages][zero 2K][bars]
// TMEM: [0, 384) the blocks' L and dw buffers (UnitBufs); O_(j, tile parity) at
// [384 + 32 (2 j + parity)).  o_full: kDxOFull barriers, as in the forward's deslice (the
// warpgroup that drains tile t has not waited for tile t - 2; it has seen the logits of a block
// at most three back, so the products four before that: tile t - 7).
// =========================================================================================
constexpr int kDxThreads = 512, kDxWGs = 3, kDxOFull = 8;
template <bool split, bool kComb = false>
__global__ void __launch_bounds__(kDxThreads, 1)
    k_bwd_dx_tc(const __grid_constant__ CUtensorMap xmap, const __grid_constant__ CUtensorMap vmap,
                const __grid_constant__ CUtensorMap pmap, const __grid_constant__ CUtensorMap dmap,
                const __grid_constant__ CUtensorMap fmap, const uint8_t* __restrict__ wimg,
                const uint8_t* __restrict__ timg, const uint8_t* __restrict__ timg2,
                const uint8_t* __restrict__ wtimg, __nv_bfloat16* __restrict__ dx, int64_t N, int64_t Np, int H,
                int Gi, int g0, int G, int splits, int hilo, int accumulate, uint32_t* status) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  constexpr uint32_t kStg = kBStage + (kComb ? kXBytes : 0u);  // x | v | px | dpx [| fx]
  const uint32_t wbytes = (uint32_t)G * (hilo ? kWRow : 96);
  uint8_t* s_w = smem;
  uint8_t* s_t = s_w + wbytes;
  uint8_t* s_t2 = s_t + (uint32_t)G * 96;
  uint8_t* s_wt = s_t2 + (kComb ? (uint32_t)G * 96 : 0u);
  uint8_t* s_st = s_wt + (uint32_t)G * 64;
  uint8_t* s_zero = s_st + kDxStages * kStg;
  uint64_t* bars = reinterpret_cast<uint64_t*>(s_zero + kPxZero);
  uint64_t* wz_full = bars;
  uint64_t* x_full = bars + 1;
  uint64_t* x_empty = x_full + kDxStages;
  uint64_t* s_full = x_empty + kDxStages;
  using Bufs = UnitBufs<false>;
  uint64_t* p_ready = s_full + Bufs::kL;  // [L buffer][half of the unit]
  uint64_t* pv_done = p_ready + 2 * Bufs::kL;
  uint64_t* dw_free = pv_done + Bufs::kL;
  uint64_t* o_full = dw_free + Bufs::kD;
  uint64_t* o_free = o_full + kDxOFull;
  uint64_t* drain = o_free + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain + 3);
  Abort* ab = reinterpret_cast<Abort*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const Work wk = work_of(N, splits, blockIdx.x, blockIdx.y);
  const int64_t b = wk.bh / H;
  const int h = (int)(wk.bh % H);
  const int nch = G / 64;
  const int total = wk.ntiles * nch;
  constexpr uint32_t kO = 384u;
  constexpr uint32_t kVOff = kXBytes, kPOff = 2 * kXBytes, kDOff = 2 * kXBytes + kPxBytes;

  if (threadIdx.x == 0) {
    mbar_init(wz_full, 1);
    for (int s = 0; s < kDxStages; s++) {
      mbar_init(&x_full[s], 1);
      mbar_init(&x_empty[s], 2);  // logits and dw issuers
    }
    for (int i = 0; i < Bufs::kL; i++) {
      mbar_init(&s_full[i], 2);  // logits and dw
      mbar_init(&p_ready[2 * i], 4);
      mbar_init(&p_ready[2 * i + 1], 4);
      mbar_init(&pv_done[i], 1);
    }
    for (int i = 0; i < Bufs::kD; i++) mbar_init(&dw_free[i], 4);
    for (int i = 0; i < kDxOFull; i++) mbar_init(&o_full[i], 1);
    for (int i = 0; i < 2; i++) mbar_init(&o_free[i], 4);
    for (int i = 0; i < 3; i++) mbar_init(&drain[i], 1);
    ab->flag = 0;
    fence_mbar_init();
  }
  zero_smem(s_zero, kPxZero);
  fence_proxy_async_smem();
  if (warp == 1) tmem_alloc(tmem_slot, 512);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  grid_trigger();
  grid_wait(wimg, timg, timg2, wtimg, dx);

  if (warp == 0) {
    if (lane == 0 && wk.ntiles > 0) {
      prefetch_tmap(&xmap);
      prefetch_tmap(&vmap);
      prefetch_tmap(&pmap);
      prefetch_tmap(&dmap);
      if (kComb) prefetch_tmap(&fmap);
      mbar_expect_tx(wz_full, wbytes + (uint32_t)G * 96 * (kComb ? 2u : 1u) + (uint32_t)G * 64);
      load_slots(s_w, wimg + (size_t)h * Gi * kWRow, Gi, g0, G, hilo, wz_full);
      load_slots(s_t, timg + (size_t)wk.bh * Gi * kWRow, Gi, g0, G, false, wz_full);
      if (kComb) load_slots(s_t2, timg2 + (size_t)wk.bh * Gi * kWRow, Gi, g0, G, false, wz_full);
      load_images(s_wt, wtimg + (size_t)h * Gi * 128 + (size_t)g0 * 64, (uint32_t)G * 64, wz_full);
      int i = 0;
      for (; i < wk.ntiles; i++) {
        const int s = i % kDxStages;
        if (i >= kDxStages && !mbar_wait(&x_empty[s], (uint32_t)(((i / kDxStages) - 1) & 1), ab, status)) break;
        uint8_t* st = s_st + s * kStg;
        const int n0 = (int)((wk.tile0 + i) * kTile);
        mbar_expect_tx(&x_full[s], kStg);
        tma_load_3d(st, &xmap, h * kD, n0, (int)b, &x_full[s]);
        tma_load_3d(st + kVOff, &vmap, h * kD, n0, (int)b, &x_full[s]);
        tma_load_2d(st + kPOff, &pmap, 0, (int)(wk.bh * Np + n0), &x_full[s]);
        tma_load_2d(st + kDOff, &dmap, 0, (int)(wk.bh * Np + n0), &x_full[s]);
        if (kComb) tma_load_3d(st + kBStage, &fmap, h * kD, n0, (int)b, &x_full[s]);
      }
      for (int j = (i > kDxStages ? i - kDxStages : 0); j < i; j++)
        mbar_wait(&x_full[j % kDxStages], (uint32_t)((j / kDxStages) & 1), ab, nullptr, kWaitNs);
      mbar_wait(wz_full, 0, ab, nullptr, kWaitNs);
    }
  } else if (warp == 1 || warp == 2) {
    // ------------------------------ logits (warp 1) and dw (warp 2) issuers ------------------------------
    if (wk.ntiles > 0) {
      const uint32_t w0 = sdesc_lo(smem_u32(s_w), 16), t0 = sdesc_lo(smem_u32(s_t), 16), t20 = sdesc_lo(smem_u32(s_t2), 16);
      const uint32_t sz = smem_u32(s_zero), ext = (uint32_t)G * 4;
      bool ok = mbar_wait_w(wz_full, 0, ab, status);
      Ring<kDxStages> stg;
      Ring<Bufs::kL> sb;
      Ring<Bufs::kD> db;
      for (int i = 0, q = 0; ok && i < wk.ntiles; i++, stg.next()) {
        if (!(ok = mbar_wait_w(&x_full[stg.i], stg.pass, ab, status))) break;
        const uint32_t st = smem_u32(s_st + stg.i * kStg);
        const uint32_t x = sdesc_lo(st, 16), v = x + kVOff / 16, f = x + kBStage / 16;
        const uint32_t px = px_lo(st + (warp == 1 ? kPOff : kDOff), sz);
        uint32_t r = 0, e = ext;  // the chunk's rows in the 64-byte and 32-byte images, in 16 bytes
#pragma unroll 1
        for (int c = 0; c < nch; c++, q++, sb.next(), db.next(), r += 64 * 4, e += 64 * 2) {
          // L: the products of the unit kL back; dw: loaded by the unit kD back
          if (q >= (warp == 1 ? Bufs::kL : Bufs::kD) &&
              !(ok = mbar_wait_w(warp == 1 ? &pv_done[sb.i] : &dw_free[db.i], (warp == 1 ? sb.pass : db.pass) ^ 1u, ab,
                                 status)))
            break;
          tc_fence_after();
          const uint32_t tL = tmem + (uint32_t)sb.i * 64, tD = tmem + Bufs::kDCol + (uint32_t)db.i * 64;
          if (warp == 1) {
            issue_dot64<false, kHiPx, kHi32>(tL, x, w0 + r, px, w0 + e, hilo ? w0 + (uint32_t)G * 6 + r : 0u);
          } else if (kComb) {
            // As in the slot pass: the deslice's chain without an extra block, the slice's
            // extra block against delta's rows (dS - delta in one K step).
            issue_dot64<false, 0, 0>(tD, v, t0 + r, 0u, 0u, 0u);
            issue_dot64<false, kHiPx, kHi32>(tD, f, t20 + r, px, t20 + e, 0u, 1u);
          } else {
            issue_dot64<false, kHiPx, kHi32>(tD, v, t0 + r, px, t0 + e, 0u);
          }
          mma_commit_w(&s_full[sb.i]);
        }
        mma_commit_w(&x_empty[stg.i]);
      }
      mma_commit_w(&drain[warp - 1]);
      mbar_wait_w(&drain[warp - 1], 0, ab, nullptr, kWaitNs);
    }
  } else if (warp == 3) {
    // ------------------------------ product issuer ------------------------------
    // K-steps [2 j, 2 j + 2) of a 64-slot chunk into O_j.
    if (wk.ntiles > 0) {
      constexpr uint32_t idesc = idesc_bf16(128, kD, false, false);
      const uint32_t wt0 = sdesc_lo(smem_u32(s_wt), 16);
      bool ok = mbar_wait_w(wz_full, 0, ab, status);
      Ring<Bufs::kL> sb;
      for (int i = 0; ok && i < wk.ntiles; i++) {
        const int ob = i & 1;
        if (i >= 2 && !(ok = mbar_wait_w(&o_free[ob], (uint32_t)(((i >> 1) - 1) & 1), ab, status))) break;
        uint32_t wt = wt0;
#pragma unroll 1
        for (int c = 0; c < nch; c++, wt += 256, sb.next()) {
#pragma unroll
          for (int j = 0; j < 2; j++) {
            if (!(ok = mbar_wait_w(&p_ready[2 * sb.i + j], sb.pass, ab, status))) break;
            tc_fence_after();
            const uint32_t tO = tmem + kO + (uint32_t)(j * 2 + ob) * kD;
            const uint32_t tL = tmem + (uint32_t)sb.i * 64 + (uint32_t)j * 32;  // da_col(2 j)
#pragma unroll
            for (int e = 0; e < 2; e++) {
              mma_ts_w<kHi128>(tO, tL + da_col(e), wt + j * 4 + e * 2, idesc, (c > 0 || e > 0) ? 1u : 0u);
              if (split) mma_ts_w<kHi128>(tO, tL + da_col(e) + 16, wt + j * 4 + e * 2, idesc, 1u);
            }
          }
          if (!ok) break;
          mma_commit_w(&pv_done[sb.i]);
        }
        mma_commit_w(&o_full[i % kDxOFull]);
      }
      mma_commit_w(&drain[2]);
      mbar_wait_w(&drain[2], 0, ab, nullptr, kWaitNs);
    }
  } else {
    const int wg = (warp - kSoftmaxWarp0) >> 2;
    const int wq = warp & 3;
    const int r = wq * 32 + lane;
    const uint32_t lane_addr = (uint32_t)(wq * 32) << 16;
    bool ok = true;
    auto epilogue = [&](int t) -> bool {
      const int ob = t & 1;
      if (!mbar_wait(&o_full[t % kDxOFull], (uint32_t)((t / kDxOFull) & 1), ab, status)) return false;
      tc_fence_after();
      uint32_t o0[32], o1[32];
      tmem_ld32(tmem + lane_addr + kO + (uint32_t)ob * kD, o0);
      tmem_ld32(tmem + lane_addr + kO + (uint32_t)(2 + ob) * kD, o1);
      tmem_wait_ld2(o0, o1);
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&o_free[ob]);
      const int64_t n = (wk.tile0 + t) * kTile + r;
      if (n < N) {
        uint4* dst = reinterpret_cast<uint4*>(dx + ((b * N + n) * H + h) * kD);
        float add[kD];
#pragma unroll
        for (int k = 0; k < kD; k++) add[k] = 0.f;
        if (accumulate) {
#pragma unroll
          for (int k = 0; k < 4; k++) {
            const uint4 q4 = dst[k];
            const uint32_t w[4] = {q4.x, q4.y, q4.z, q4.w};
#pragma unroll
            for (int e = 0; e < 4; e++) {
              add[8 * k + 2 * e] = __uint_as_float(w[e] << 16);
              add[8 * k + 2 * e + 1] = __uint_as_float(w[e] & 0xFFFF0000u);
            }
          }
        }
#pragma unroll
        for (int k = 0; k < 4; k++) {
          uint32_t w[4];
#pragma unroll
          for (int e = 0; e < 4; e++) {
            const int c0 = 8 * k + 2 * e;
            w[e] = pack_bf16(fmaf(__uint_as_float(o0[c0]) + __uint_as_float(o1[c0]), kLn2, add[c0]),
                             fmaf(__uint_as_float(o0[c0 + 1]) + __uint_as_float(o1[c0 + 1]), kLn2, add[c0 + 1]));
          }
          dst[k] = make_uint4(w[0], w[1], w[2], w[3]);
        }
      }
      return true;
    };
    BlockPos pos(wg, nch);
    for (int q = wg; ok && q < total; q += kDxWGs, pos.step(kDxWGs, nch)) {
      const int i = pos.i, c = pos.c;
      const int bb = q % Bufs::kL, bd = q % Bufs::kD;
      if (!(ok = mbar_wait(&s_full[bb], (uint32_t)((q / Bufs::kL) & 1), ab, status))) break;
      tc_fence_after();
      const uint32_t tL = tmem + lane_addr + (uint32_t)bb * 64;
      const uint32_t tD = tmem + lane_addr + Bufs::kDCol + (uint32_t)bd * 64;
      float unused0 = 0.f, unused1 = 0.f;
#pragma unroll
      for (int hf = 0; hf < 2; hf++) {
        da_half<split, false, false>(tL + 32 * hf, tD + 32 * hf, unused0, unused1, [&]() {
          if (hf == 1) {
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&dw_free[bd]);
          }
        });
        tmem_wait_st();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&p_ready[2 * bb + hf]);
      }
      if (c == 0 && i > 0 && !(ok = epilogue(i - 1))) break;
    }
    if (ok && total > 0 && total % kDxWGs == wg) epilogue(wk.ntiles - 1);
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 1) tmem_dealloc(tmem, 512);
}

// ---- host side ---------------------------------------------------------------------------------

size_t smem_bwd_slot(int mode = 1) {
  const bool m3 = mode == 3;
  return 1024 + (m3 ? 3 : 2) * (size_t)kWBlockB + (m3 ? kBStages - 1 : kBStages) * (size_t)(kBStage + (m3 ? kXBytes : 0)) +
         kPxZero + 3 * kGC * 4 + 512;
}
size_t smem_bwd_dx(int G, bool hilo, bool comb = false) {
  return 1024 + (size_t)G * ((hilo ? kWRow : 96) + 96 * (comb ? 2 : 1) + 64) +
         kDxStages * (size_t)(kBStage + (comb ? kXBytes : 0)) + kPxZero + 512;
}

int bwd_slot_blocks(const Shape& s) { return s.G / kGC; }
// Point splits of the slot pass.  MODE 1 (fs_deslice_bwd) keeps dW and d z' in one accumulator
// chain a half for a CTA's whole range, and a chain of tensor-core sums drifts towards zero with
// its length, ~2^-26 relative per 16 points (d z' at B = 1, N = 262,144, H = 8, G = 1024 in 19
// splits 1.3e-5 from 64 bits, in 7 splits 3.4e-5); so a range longer than kChainTiles, whose drift
// of 5e-7 the other errors (3e-6) hide, takes more splits, up to those of whole waves.  (Whole
// waves' splits for every range: separate backward calls at B = 2, N = 4,096, H = 8, G = 256 149
// us against 132.)  The other modes flush their chains.
constexpr int kChainTiles = 4;
int bwd_slot_splits(const Shape& s, int mode) {
  const int units = (int)(s.BH() * bwd_slot_blocks(s));
  const int P = point_splits(s, units, 2);
  if (mode != 1) return P;
  const int64_t tiles = padded_n(s) / kTile;
  return (int)std::min<int64_t>(wave_splits(s, units), std::max<int64_t>(P, (tiles + kChainTiles - 1) / kChainTiles));
}

// Slot ranges.  The images of a call cover all of its slots; the rows and point passes, which
// hold images in shared memory (a rows pass W' and t with their residuals, the point pass
// W', W'^T and one T image, in fs_coupling_bwd two), run over ranges of at most so many
// slots, all with the full problem's lse, so that the weights of a range are those of the
// softmax over all G.  The sums over slots (delta, dfx, dx) add up over the ranges.  The slot
// pass holds one 128-slot block and needs no ranges.  As few ranges as fit (a range re-reads
// x and v), of equal size but for the last.
// (The separate calls' point pass holds the residual half of W' up to 512 slots: past 640,
// where it runs over ranges anyway, no range is longer, which keeps dx of a sum over many
// ranges accurate.)
constexpr int kBwdSlotsMax = 640, kCombSlotsMax = 256, kPointSlotsMax = 512, kRowsBothMax = 512;
struct SlotRanges {
  int n, size;
};
SlotRanges slot_ranges(int Gp, int most) {
  const int n = (Gp + most - 1) / most;
  return {n, (Gp / kGC + n - 1) / n * kGC};
}

// fs_coupling_bwd: one rows pass for both parts where the images of both t fit (512 slots).
// Ranges cut to fit would round dfx to bf16 once more a range and run the epilogue again, so
// longer ranges (513 to 640 slots) keep a pass for each part.
bool rows_both(const Shape& s) { return slot_ranges(s.G, kBwdSlotsMax).size <= kRowsBothMax; }

SlotRanges point_ranges(int Gp, bool comb) {
  return slot_ranges(Gp, comb ? kCombSlotsMax : (Gp <= kBwdSlotsMax ? kBwdSlotsMax : kPointSlotsMax));
}

// The backward forms every weight with split products whatever the forward's
// arithmetic: its lse comes from split products (recomputed when the forward's
// did not), and weights from bf16 logits would not sum to one against it; the
// excess would bias the gradients that are sums of cancelling terms (dbias, dtau).
Shape split_shape(const Shape& s) {
  Shape r = s;
  r.dot = FS_DOT_BF16X2;
  return r;
}
// The shape the passes see: split products, whole 128-slot blocks.
Shape pass_shape(const Shape& s0) { return tc_padded(split_shape(s0)); }

enum BwdKind { kDesliceBwd = 1, kSliceBwd = 2, kCouplingBwd = 3 };

// Workspace layout of one tensor-core backward call (offsets from the tc region).
struct BwdLayout {
  size_t wimg, wtimg, timg, timg2, zimg, px, dpx, delta, delta_d, wds, ds, dtp, part, sl_part, sl_wsum, total;
};
BwdLayout bwd_layout(const Shape& s0, BwdKind kind) {
  BwdLayout L{};
  size_t off = 0;
  auto take = [&](size_t bytes) {
    const size_t o = off;
    off = align_up(off + bytes, 256);
    return o;
  };
  const Shape s = pass_shape(s0);
  const size_t BHG = (size_t)s.BH() * s.G;
  const size_t pts = (size_t)s.BH() * s.N;
  const int P = bwd_slot_splits(s, kind == kDesliceBwd ? 1 : 2), R = bwd_slot_blocks(s);
  const bool comb = kind == kCouplingBwd;
  L.wimg = take(w_image_bytes(s));
  L.wtimg = take((size_t)s.H * s.G * 128);
  L.timg = take(BHG * kWRow);
  L.timg2 = take(comb ? BHG * kWRow : 0);
  L.zimg = take(BHG * 128);
  L.px = take(px_bytes(s));
  L.dpx = take(px_bytes(s));
  L.delta = take(pts * sizeof(float));
  const bool both = comb && rows_both(s);
  L.delta_d = take(comb && !both ? pts * sizeof(float) : 0);
  L.wds = take(kind != kDesliceBwd ? (both ? 3 : 2) * pts * sizeof(float) : 0);
  L.ds = take(BHG * sizeof(float));
  L.dtp = take((size_t)s.BH() * P * R * sizeof(float));
  // (rows_both: the second zimg, whose last reader is done when the slot pass writes here)
  L.part = take((size_t)P * BHG * (kind == kDesliceBwd ? 2 * kD + 2 : kD + 2) * sizeof(float));
  // d z' of the coupling through the forward's slice
  const bool via_slice = comb && tc_forward_supported(split_shape(s0));
  L.sl_part = take(via_slice ? tc_slice_partials_bytes(split_shape(s0)) : 0);
  L.sl_wsum = take(via_slice ? (size_t)s.BH() * s0.G * sizeof(float) : 0);
  L.total = off;
  return L;
}

// The passes of a call on its layout.
struct BwdCall {
  const Shape &s0, s;  // the caller's shape; the padded one
  const BwdLayout L;
  uint8_t* ws;
  uint32_t* status;
  cudaStream_t st;
  BwdCall(const Shape& s0_, BwdKind kind, void* w, uint32_t* status_, cudaStream_t st_)
      : s0(s0_), s(pass_shape(s0_)), L(bwd_layout(s0_, kind)), ws(static_cast<uint8_t*>(w)), status(status_), st(st_) {}
  float* f(size_t off) const { return reinterpret_cast<float*>(ws + off); }

  // delta and, mode 2, dfx and the sums of w dS, over the slot ranges; zimg holds t.
  // Mode 3: both parts (v = fx, v2 = dO; zimg holds z', the part region dU).
  cudaError_t rows(int mode, const void* x, const void* v, const void* v2, void* dfx, float* delta) const {
    const SlotRanges r = slot_ranges(s.G, kBwdSlotsMax);
    for (int k = 0; k < r.n; k++) {
      const int g0 = k * r.size;
      Shape sr = s;
      sr.G = std::min(r.size, s.G - g0);
      if (cudaError_t e = tc_rows_bwd(sr, s.G, g0, mode, x, ws + L.wimg, ws + L.zimg, ws + L.part, ws + L.px, v, v2, dfx, delta,
                                      mode != 1 ? f(L.wds) : nullptr, f(L.ds), k > 0 ? 1 : 0, status, st))
        return e;
    }
    return cudaSuccess;
  }
  // u = dz / (S + eps) and c as images (T at `timg`, Z layout at `zimg`) and ds.
  cudaError_t images_us(const float* z, const float* wsum, const float* dz, size_t timg, size_t zimg) const {
    return launch(k_prep_us, dim3((unsigned)(s.G / 64), (unsigned)s.BH()), dim3(256), 0, st, z, wsum, dz, ws + timg,
                  ws + zimg, f(L.ds), s0.G, s.G, s.eps);
  }
  // delta's point rows from delta (+ delta2) (+ the sums of w dS).
  cudaError_t delta_rows(const float* delta, const float* delta2, const float* wds, int nwds) const {
    const int64_t n = s.BH() * padded_n(s);
    return launch(k_prep_dpx, dim3((unsigned)((n + 255) / 256)), dim3(256), 0, st, delta, delta2, wds, nwds,
                  reinterpret_cast<uint4*>(ws + L.dpx), s.BH(), s.N, padded_n(s));
  }
  // The slot pass over all slots (v, f: the deslice's and the slice's points of MODE 3).
  template <int MODE>
  cudaError_t slot(const void* x, const void* v, const void* f3) const {
    CUtensorMap xmap, vmap, pmap, dmap, fmap;
    if (!make_maps(x, v, f3, &xmap, &vmap, &pmap, &dmap, &fmap)) return cudaErrorInvalidValue;
    const size_t sm = smem_bwd_slot(MODE);
    const auto kernel = k_bwd_slot_tc<MODE, true>;
    if (cudaError_t e = set_smem(kernel, sm)) return e;
    const int P = bwd_slot_splits(s, MODE);
    return launch(kernel, dim3((unsigned)bwd_slot_blocks(s), (unsigned)P, (unsigned)s.BH()), dim3(kThreads), sm, st,
                  xmap, vmap, pmap, dmap, fmap, ws + L.wimg, ws + L.timg, ws + L.timg2, f(L.part), f(L.dtp), s.N,
                  padded_n(s), s.H, s.G, P, status);
  }
  // dW, dbias, dtau (and d z' into dzp) from the slot pass's partials.
  cudaError_t reduce(const float* tau, float* dzp, float* dW, float* db, float* dtau, int accumulate) const {
    const int P = bwd_slot_splits(s, dzp ? 1 : 2);
    return reduce_bwd(s0, P, f(L.part), s.G, dzp ? 2 * kD + 2 : kD + 2, tau, dzp, dW, db, dtau, f(L.dtp),
                      (int64_t)P * bwd_slot_blocks(s), accumulate, st);
  }
  // dx over the slot ranges.
  template <bool kComb>
  cudaError_t point(const void* x, const void* v, const void* f3, void* dx, int accumulate) const {
    CUtensorMap xmap, vmap, pmap, dmap, fmap;
    if (!make_maps(x, v, f3, &xmap, &vmap, &pmap, &dmap, &fmap)) return cudaErrorInvalidValue;
    const SlotRanges r = point_ranges(s.G, kComb);
    const bool hilo = smem_bwd_dx(r.size, true, kComb) <= kMaxSmem;
    const size_t sm = smem_bwd_dx(r.size, hilo, kComb);
    if (sm > kMaxSmem) return cudaErrorInvalidValue;
    const auto kernel = k_bwd_dx_tc<true, kComb>;
    if (cudaError_t e = set_smem(kernel, sm)) return e;
    const int P = point_splits(s, (int)s.BH(), r.size / 64);
    for (int k = 0; k < r.n; k++) {
      const int g0 = k * r.size;
      if (cudaError_t e = launch(kernel, dim3((unsigned)P, (unsigned)s.BH()), dim3(kDxThreads), sm, st, xmap, vmap, pmap,
                                 dmap, fmap, ws + L.wimg, ws + L.timg, ws + L.timg2, ws + L.wtimg,
                                 static_cast<__nv_bfloat16*>(dx), s.N, padded_n(s), s.H, s.G, g0,
                                 std::min(r.size, s.G - g0), P, hilo ? 1 : 0, (accumulate || k > 0) ? 1 : 0,
                                 status)) return e;
    }
    return cudaSuccess;
  }
  bool make_maps(const void* x, const void* v, const void* f3, CUtensorMap* xmap, CUtensorMap* vmap, CUtensorMap* pmap,
                 CUtensorMap* dmap, CUtensorMap* fmap) const {
    const int64_t Np = padded_n(s);
    return make_point_map(xmap, x, s, kD, CU_TENSOR_MAP_SWIZZLE_64B) &&
           make_point_map(vmap, v, s, kD, CU_TENSOR_MAP_SWIZZLE_64B) && make_px_map(pmap, ws + L.px, s.BH(), Np) &&
           make_px_map(dmap, ws + L.dpx, s.BH(), Np) &&
           make_point_map(fmap, f3 ? f3 : x, s, kD, CU_TENSOR_MAP_SWIZZLE_64B);
  }
};

#define FS_TRY(call)                                  \
  do {                                                \
    if (cudaError_t e_ = (call)) return e_;           \
  } while (0)

}  // namespace

// A single point (N = 1) takes the fp32 SIMT backward: every token is then that
// point's fx times S/(S + eps), so the slice's gradients are O(eps) and come from
// cancelling terms of size |dz||fx|/(S + eps) that split bf16 products resolve only
// to ~2^-17 of that size.
bool tc_backward_supported(const Shape& s0) {
  if (s0.dtype != FS_BF16 || s0.d != kD || s0.N < 2 || s0.G > 4096) return false;
  Shape s = pass_shape(s0);
  s.G = slot_ranges(s.G, kBwdSlotsMax).size;
  return tc_forward_supported(s) && smem_bwd_dx(s.G, false) <= kMaxSmem &&
         tc_rows_smem(s) <= kMaxSmem;
}

size_t tc_backward_bytes(const Shape& s, int mode) {
  return tc_backward_supported(s) ? bwd_layout(s, mode == 1 ? kDesliceBwd : kSliceBwd).total : 0;
}

int tc_backward_launch_count(const Shape& s, int mode) {
  const int G = pass_shape(s).G;
  // prep, delta's rows, slot, reductions; rows and point per range; mode 2 also u's images
  return 4 + slot_ranges(G, kBwdSlotsMax).n + point_ranges(G, false).n + (mode == 2 ? 1 : 0);
}

// dz' (the slot pass, MODE 1), dW, dbias, dtau, dx of the deslice: the rows pass forms delta,
// the slot pass the slot-owned gradients, the point pass dx.
cudaError_t tc_deslice_bwd(const Shape& s0, const void* x, const float* W, const float* bias, const float* tau,
                           const float* zp, const float* lse, const void* dout, float* dzp, void* dx, float* dW,
                           float* db, float* dtau, int accumulate, void* ws_tc, bool reset, uint32_t* status,
                           cudaStream_t st) {
  const BwdCall c(s0, kDesliceBwd, ws_tc, status, st);
  Prepare p(c.s, s0.G, tau, status, reset);
  p.weights(W, bias, c.ws + c.L.wimg);
  p.weights_t(W, c.ws + c.L.wtimg);
  p.tokens(zp, c.ws + c.L.timg, c.ws + c.L.zimg, true);
  p.rows(lse, c.ws + c.L.px);
  FS_TRY(p.run(st));
  FS_TRY(c.rows(1, x, dout, nullptr, nullptr, c.f(c.L.delta)));
  FS_TRY(c.delta_rows(c.f(c.L.delta), nullptr, nullptr, 0));
  FS_TRY(c.slot<1>(x, dout, nullptr));
  FS_TRY(c.reduce(tau, dzp, dW, db, dtau, accumulate));
  return c.point<false>(x, dout, nullptr, dx, accumulate);
}

cudaError_t tc_slice_bwd(const Shape& s0, const void* x, const void* f, const float* W, const float* bias,
                         const float* tau, const float* z, const float* wsum, const float* lse, const float* dz,
                         void* dx, void* dfx, float* dW, float* db, float* dtau, int accumulate, void* ws_tc,
                         bool reset, uint32_t* status, cudaStream_t st) {
  const BwdCall c(s0, kSliceBwd, ws_tc, status, st);
  Prepare p(c.s, s0.G, tau, status, reset);
  p.weights(W, bias, c.ws + c.L.wimg);
  p.weights_t(W, c.ws + c.L.wtimg);
  p.rows(lse, c.ws + c.L.px);
  p.clear(c.f(c.L.wds), 2 * c.s.BH() * c.s.N);
  FS_TRY(p.run(st));
  FS_TRY(c.images_us(z, wsum, dz, c.L.timg, c.L.zimg));
  FS_TRY(c.rows(2, x, f, nullptr, dfx, c.f(c.L.delta)));
  FS_TRY(c.delta_rows(c.f(c.L.delta), nullptr, c.f(c.L.wds), 2));
  FS_TRY(c.slot<2>(x, f, nullptr));
  FS_TRY(c.reduce(tau, nullptr, dW, db, dtau, accumulate));
  return c.point<false>(x, f, nullptr, dx, accumulate);
}

size_t tc_coupling_bwd_bytes(const Shape& s) {
  return tc_backward_supported(s) ? bwd_layout(s, kCouplingBwd).total : 0;
}

int tc_coupling_bwd_launch_count(const Shape& s) {
  const int G = pass_shape(s).G, n = slot_ranges(G, kBwdSlotsMax).n;
  // prep; d z' (slice or slot pass, reduction), the mix backward, u's images; delta's rows,
  // slot, reductions; the rows passes and the point pass per range
  return 1 + 2 + 1 + 1 + 3 + (rows_both(pass_shape(s)) ? 1 : 2) * n + point_ranges(G, true).n;
}

// The coupling's backward in one call (fs_coupling_bwd).  The deslice's and the
// slice's da share the weights, so their slot-owned and point-owned products can be
// formed once from da_D + da_S; what has to come first is d z' (it feeds the mix
// backward, and so dU, dS and the slice's part):
//   1. d z' = sum_n w_ng dO_n: the forward's slice with dO for fx (its unnormalised
//      numerators) where the forward's kernels take the shape, else the slot pass in
//      mode 0 (the weights alone);
//   2. the mix backward and the images of dU | dS;
//   3. the rows pass in mode 3: delta_D + delta_S, dfx, the sum_g w dS partials (past 512
//      slots a range: in mode 1 for the deslice part, first, and here in mode 2);
//   4. delta + sum_g w dS into the point rows;
//   5. the slot pass in mode 3: dW, dbias, dtau of da_D + da_S;
//   6. the point pass for dx.
cudaError_t tc_coupling_bwd(const Shape& s0, const void* x, const void* f, const void* dout, const float* W,
                            const float* bias, const float* tau, const float* M, const float* z, const float* wsum,
                            const float* zp, const float* lse, float* dzp, float* dz, float* dM, void* dx, void* dfx,
                            float* dW, float* db, float* dtau, int accumulate, void* ws_tc, bool reset,
                            uint32_t* status, cudaStream_t st) {
  const BwdCall c(s0, kCouplingBwd, ws_tc, status, st);
  const BwdLayout& L = c.L;
  Prepare p(c.s, s0.G, tau, status, reset);
  p.weights(W, bias, c.ws + L.wimg);
  p.weights_t(W, c.ws + L.wtimg);
  p.tokens(zp, c.ws + L.timg, c.ws + L.zimg, true);
  p.rows(lse, c.ws + L.px);
  const bool both = rows_both(c.s);
  const int nwds = both ? 3 : 2;
  p.clear(c.f(L.wds), nwds * c.s.BH() * c.s.N);
  FS_TRY(p.run(st));
  if (!both) FS_TRY(c.rows(1, x, dout, nullptr, nullptr, c.f(L.delta_d)));
  if (tc_forward_supported(split_shape(s0))) {
    FS_TRY(run_slice(c.s, s0.G, x, dout, nullptr, nullptr, c.ws + L.wimg, c.ws + L.px, dzp, c.f(L.sl_wsum), 0,
                     c.f(L.sl_part), status, st));
  } else {
    FS_TRY(c.slot<0>(x, dout, nullptr));
    FS_TRY(simt_reduce_dzp(s0, bwd_slot_splits(c.s, 0), c.f(L.part), c.s.G, kD, dzp, st));
  }
  FS_TRY(mix_bwd(s0, M, z, dzp, dz, dM, st));
  FS_TRY(c.images_us(z, wsum, dz, L.timg2, both ? L.part : L.zimg));
  FS_TRY(c.rows(both ? 3 : 2, x, f, dout, dfx, c.f(L.delta)));
  FS_TRY(c.delta_rows(c.f(L.delta), both ? nullptr : c.f(L.delta_d), c.f(L.wds), nwds));
  FS_TRY(c.slot<3>(x, dout, f));
  FS_TRY(c.reduce(tau, nullptr, dW, db, dtau, accumulate));
  return c.point<true>(x, dout, f, dx, accumulate);
}

}  // namespace fs
