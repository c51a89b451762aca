// Tensor-core forward path on sm_103a (tcgen05 + TMEM + TMA), and the rows pass
// of the backward (the deslice kernel in modes 1 and 2, see k_deslice).
//
// Inputs: bf16 point tensors as they are; fp32 point tensors split beforehand
// into bf16 hi and residual tensors (k_prep), with the residual products
// added in the X3 instantiations.  G is padded to whole 128-slot blocks whose
// padding slots carry weight 0.
//
// The three streaming passes of the paper's G-blocked family (Appendix G.1):
//   k_stats   : per point and head, lse_n = log sum_g exp(a_ng)        (point-owned)
//   k_slice   : per slot, U_g = sum_n w_ng f_n and S_g = sum_n w_ng     (slot-owned,
//               split over points; the partials are summed in a fixed order after)
//   k_deslice : per point, out_n = sum_g w_ng z'_g                      (point-owned)
// w is recomputed tile by tile in every pass and never leaves the SM.
//
// Logits.  A 128-point x 128-slot block of base-2 logits a2 = a * log2(e) is one
// tcgen05.mma chain with K = 48:
//   point side [ x (32 bf16) | 1, 1, -lse2 (three bf16 parts), 0 ... ]  (stats: 1, 1, 0 ...)
//   slot side  [ W*log2e/tau (32) | b'_hi, b'_lo, 1, 1, 1, 0 ... ]  (b' = bias*log2e/tau
//                                                                 in two bf16 halves)
// The point-major passes (stats, deslice) put points on the MMA's M (TMEM lane
// = point); the slice swaps the operands, so its TMEM lane is a slot and its
// column a point.  In the slice and the deslice the point side's extra block is
// [1, 1, -lse2 in three parts, 0 ...], so the accumulator holds a2 - lse2, the
// log2 of the slice weight itself.  The stats pass writes these 16-byte rows per
// point to memory and the later passes load them by TMA with each tile: no
// thread writes a tensor-core operand per tile (that would cost a generic ->
// async proxy fence per tile).
//
// Products.  The bf16 weights are written back into the S buffer they came
// from and feed the second MMA as its TMEM A operand: P x Z' in the deslice
// (M = points, K = slots, N = 32 channels), E x [F | 1] in the slice (M =
// slots, K = points, N = 48: 32 channels and a ones column for the weight sums).
//
// Issue.  Each MMA-issuing role is a whole converged warp in which one elected
// lane issues (a lone lane in a divergent branch issues several times slower).
// Warp 1 issues the logits; warps 2 and 3 issue the
// products into accumulators of their own, which are summed in a fixed order,
// so the result is deterministic.
//
// CTA: warp 0 TMA producer, warps 1..3 MMA issuers, warps 4 and up softmax warpgroups
// (two to four) that take blocks in turn (so they run out of phase);
// a thread owns one TMEM lane (tcgen05.ld/st 32x32b).  Every wait is bounded
// (2 s and 2,000 polls): a wait that gives up writes FS_ERR_TIMEOUT to the status word, the CTA
// drains its copies and MMAs, frees TMEM and exits.
//
// Shared-memory operand layouts (all bases 1024-byte aligned):
//   x tile          K-major, 64 B rows, 64B swizzle (TMA)        128 points x 32
//   constant extra  K-major, 32 B rows, 32B swizzle              128 rows x 16
//   point extra     K-major, no swizzle: core matrices of 8 rows x 16 B, the
//                   k = 0..7 half from memory (TMA), the k = 8..15 half zero
//   W image         K-major, 64 B rows, 64B swizzle, then its 32 B extra rows
//   Z' image        K-major rows = channels, 128 B rows, 128B swizzle
//   [F | 1]         MN-major, three 16-channel blocks, 32B swizzle (TMA)
#include "fs_tc_common.cuh"

namespace fs {
namespace {

using namespace tc;

// =========================================================================================
// Deslice: out_n = sum_g w_ng z'_g.
// smem: [W img G*96][Z' img G*64][stages: x | point extra (TMA half, zero half)][barriers]
// TMEM: S buffers [0, 384); P x Z' accumulators O_0 [384, 448), O_1 [448, 512), each
// double-buffered by tile parity (MODE 3: 64 columns wide and single).  Block q (tile q / nb, slot block q % nb) uses S buffer
// q % 3; a softmax warpgroup writes the bf16 weights of its 128 slots, packed in pairs,
// into columns [0, 64) of the same buffer; warp 2 + j turns slots [64 j, 64 j + 64) of every
// block into products (K-steps [4 j, 4 j + 4)) accumulated in O_j.
//
// What bounds it is each buffer's cycle logits -> exponentials -> products -> logits: a
// block takes ~760 clocks where its exponentials need 512 of MUFU and a loop of loads,
// exponentials and stores alone runs at 620 (synchronisation included, measured).  The
// forward with single-level products (MODE 0, !PS) therefore runs three softmax warpgroups
// (512 threads), one per S buffer, and hands each 64-slot half of the weights over as soon as
// it is written, so that its products run under the other half's exponentials (N = 262,144,
// H = 8, call: G = 1024 373 -> 355 us, G = 512 232 -> 211, G = 256 133 -> 118, against four
// warpgroups on half rows).  Weights in a buffer of their own with two S buffers, which frees
// S before the exponentials, was slower (375 with three warpgroups, 411 with four).  The split
// products (all halves handed over the same way) run three warpgroups as well: fp32 deslice
// call at B = 1, N = 262,144, H = 8, G = 512 410 us with two, 404 with three, 372 with 32
// columns at a time in registers.  MODE 2 keeps two (its scratch holds two partial sums of
// w dS a point), warpgroup q % 2 taking block q.
//
// The same pass serves the backward (Sec. 3.3): with R_n = sum_g w_ng t_g,
//   MODE 1 (deslice backward, t = z', v = dO): delta_n = dO_n . R_n (fp32);
//   MODE 2 (slice backward, t = dU, v = fx): dfx_n = R_n (bf16, into out) and
//     delta_n = fx_n . R_n + sum_g w_ng dS_g.  The second sum is formed by the
//     softmax warpgroups from the fp32 weights; each warpgroup adds its own
//     partial per point to wds[wg][bh][n] (cleared beforehand) and the consumer adds them;
//   MODE 3, both at once (the whole coupling's backward; z' in zimg, dU in zimg2): the
//     weights are formed once.  delta_n = dO_n . R_n + fx_n . R2_n, dfx_n = R2_n.  z' and dU
//     rows of 64 slots lie one after the other, so one MMA (N = 64) multiplies both; warp 3
//     issues them all, slot half j of every block into O_j as in the other modes: a chain of
//     tensor-core sums drifts towards zero with its length, and one chain of all slots, with an
//     accumulator per tile parity, left sum_g da_ng at 4.0e-6 of delta_n against 1.7e-6
//     (G = 512) and dbias and dW 5% further off.  Two chains leave no columns for a second tile,
//     so a tile is drained before the next one's products (whole backward at B = 2, N = 131,072,
//     H = 8: G = 512 1727 -> 1740 us, 256 933 -> 936, 64 574 -> 575).  The images take 416 B a
//     slot, so at 512 slots one x stage is left; three are no faster (G = 256: 1037 us with
//     three, 1042 with one).  What bounds it is the softmax warps: without the w dS sums the whole
//     backward took 7% less, without the epilogue's loads and stores 6%, without two of three
//     products 2%.  Whole backward at B = 2, N = 131,072, H = 8, G = 512: 2165 us with a MODE
//     1 and a MODE 2 pass, 1849 with this one.
// The pass covers slots [g0, g0 + G) of images of Gi slots.  accumulate (MODES 1 to 3, and
// MODE 0 with X3): a later range of the slots, whose contributions to delta and dfx (to the
// fp32 out) are added to those of the earlier ranges.
// PS (split products): the weights and t as bf16 hi + lo halves, P t = Phi thi +
// Plo thi + Phi tlo; the image then holds t's residual half after its bf16 half.
// The split weights of slot half j (slots [64 j, 64 j + 64) of the block) go to columns
// [64 j, 64 j + 64) of the S buffer: per 32 slots the hi pairs, then the lo pairs.
// =========================================================================================
constexpr uint32_t kDStage = kXBytes + 2 * kPxBytes;  // x tile, point extra (both halves)

// X3 (fp32 inputs, MODE 0 with PS): each stage also holds x's residual tile
// (xrmap), the logits add x_r W'_hi, and out is fp32.
template <int MODE>
constexpr bool desl_wg3() { return MODE != 2; }
constexpr int kDesl3Threads = 512;
// Barriers of completed tiles.  With three warpgroups the one that drains tile t has not
// waited for tile t - 2 (the accumulator's previous tile), and a parity wait on a barrier
// two phases behind would pass at once; what it has seen (the logits of a block at most three
// blocks back, so the products three blocks before that: tile t - 5) covers tile t - 8.
constexpr int kOFull = 8;
template <int MODE, bool PS, bool X3 = false>
__global__ void __launch_bounds__(desl_wg3<MODE>() ? kDesl3Threads : kThreads, 1)
    k_deslice(const __grid_constant__ CUtensorMap xmap, const __grid_constant__ CUtensorMap pmap,
              const __grid_constant__ CUtensorMap xrmap,
              const uint8_t* __restrict__ wimg, const uint8_t* __restrict__ zimg, const uint8_t* __restrict__ zimg2,
              __nv_bfloat16* __restrict__ out, const __nv_bfloat16* __restrict__ v,
              const __nv_bfloat16* __restrict__ v2, float* __restrict__ delta, float* __restrict__ wds,
              const float* __restrict__ dS, int64_t N, int64_t Np, int H, int Gi, int g0, int G, int splits,
              int hilo, uint32_t zstride, int nst, int accumulate, uint32_t* status) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  // hilo: the residual half of W' fits in shared memory too (K = 80 logits, as in
  // the statistics pass); else bf16 W' only (K = 48).
  const uint32_t wbytes = (uint32_t)G * (hilo ? kWRow : 96), zbytes = (uint32_t)G * (MODE == 3 ? 256 : PS ? 128 : 64);
  constexpr bool kDs = MODE == 2 || MODE == 3;
  const int ns = MODE == 3 ? nst : kStages;  // stages
  uint8_t* s_w = smem;
  uint8_t* s_z = s_w + wbytes;
  float* s_ds = reinterpret_cast<float*>(s_z + zbytes);  // kDs: dS of the G slots
  // (the stages stay 1024-byte aligned for their swizzled tiles)
  uint8_t* s_x = s_z + zbytes + (kDs ? (((uint32_t)G * 4 + 1023u) & ~1023u) : 0u);  // stage s at s_x + s * kDSt
  constexpr uint32_t kDSt = kDStage + (X3 ? kXBytes : 0u);  // stage: x | px (2 halves) [| x residual]
  uint64_t* bars = reinterpret_cast<uint64_t*>(s_x + ns * kDSt);
  uint64_t* wz_full = bars;
  uint64_t* x_full = bars + 1;
  uint64_t* x_empty = x_full + kStages;
  uint64_t* s_full = x_empty + kStages;
  constexpr bool kWG3 = desl_wg3<MODE>();
  uint64_t* p_ready = s_full + kSBuf;  // [S buffer][half]
  uint64_t* pv_done = p_ready + 2 * kSBuf;
  uint64_t* o_full = pv_done + kSBuf;
  uint64_t* o_free = o_full + kOFull;
  uint64_t* drain = o_free + 2;  // one per issuing warp
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain + 3);
  Abort* ab = reinterpret_cast<Abort*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const Work wk = work_of(N, splits, blockIdx.x, blockIdx.y);
  const int64_t b = wk.bh / H;
  const int h = (int)(wk.bh % H);
  const int nch = G / kGC;
  constexpr uint32_t kO = kSBuf * kGC;  // TMEM column base of the O accumulators
  constexpr int kWGs = kWG3 ? 3 : 2;    // softmax warpgroups
  const int total = wk.ntiles * nch;

  if (threadIdx.x == 0) {
    mbar_init(wz_full, 1);
    for (int s = 0; s < kStages; s++) {
      mbar_init(&x_full[s], 1);
      mbar_init(&x_empty[s], 1);
    }
    for (int i = 0; i < kSBuf; i++) {
      mbar_init(&s_full[i], 1);
      mbar_init(&p_ready[2 * i], 4);  // the four warps of the warpgroup that owns the block
      mbar_init(&p_ready[2 * i + 1], 4);
      mbar_init(&pv_done[i], MODE == 3 ? 1 : 2);
    }
    for (int i = 0; i < kOFull; i++) mbar_init(&o_full[i], MODE == 3 ? 1 : 2);
    for (int i = 0; i < 2; i++) mbar_init(&o_free[i], 4);
    for (int i = 0; i < 3; i++) mbar_init(&drain[i], 1);
    ab->flag = 0;
    fence_mbar_init();
  }
  for (int s = 0; s < ns; s++) zero_smem(s_x + s * kDSt + kXBytes + kPxBytes, kPxBytes);
  fence_proxy_async_smem();
  if (warp == 1) tmem_alloc(tmem_slot, 512);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  grid_trigger();
  // (The softmax warps' pointers take the zero through the row index r: seven opaque 64-bit
  // pointers cost registers that the 512-thread launch does not have.)
  const int after_wait = (int)grid_wait(wimg, zimg, zimg2, dS);
  if (kDs) {
    for (int g = threadIdx.x; g < G; g += blockDim.x) s_ds[g] = dS[wk.bh * Gi + g0 + g];
    __syncthreads();
  }

  if (warp == 0) {
    // ------------------------------ producer ------------------------------
    // (Point rows formed here from lse instead of loaded from px were slower below eight slot
    // blocks per tile: at G = 256 the call took 465 us against 425, at G = 1024 0.8% less.)
    if (lane == 0 && wk.ntiles > 0) {
      prefetch_tmap(&xmap);
      prefetch_tmap(&pmap);
      if (X3) prefetch_tmap(&xrmap);
      mbar_expect_tx(wz_full, wbytes + zbytes);
      load_slots(s_w, wimg + (size_t)h * Gi * kWRow, Gi, g0, G, hilo, wz_full);
      const uint8_t* zi = zimg + (size_t)wk.bh * zstride + (size_t)g0 * 64;
      if (MODE == 3) {
        // per 64 slots z' then t2, 32 channel rows each; all hi halves, then all lo halves
        const uint8_t* zi2 = zimg2 + (size_t)wk.bh * zstride + (size_t)g0 * 64;
        for (int hl = 0; hl < 2; hl++)
          for (int k = 0; k < G / 64; k++) {
            uint8_t* dst = s_z + (size_t)hl * G * 128 + (size_t)k * 8192;
            const size_t src = (size_t)hl * Gi * 64 + (size_t)k * 4096;
            bulk_load(dst, zi + src, 4096, wz_full);
            bulk_load(dst + 4096, zi2 + src, 4096, wz_full);
          }
      } else {
        load_images(s_z, zi, (uint32_t)G * 64, wz_full);
      }
      if (PS && MODE != 3) load_images(s_z + (uint32_t)G * 64, zi + (size_t)Gi * 64, (uint32_t)G * 64, wz_full);
      RingOf st(ns);
      int i = 0;
      for (; i < wk.ntiles; i++, st.next()) {
        if (i >= ns && !mbar_wait(&x_empty[st.i], st.pass ^ 1u, ab, status)) break;
        uint8_t* stage = s_x + st.i * kDSt;
        const int n0 = (int)((wk.tile0 + i) * kTile);
        mbar_expect_tx(&x_full[st.i], kXBytes + kPxBytes + (X3 ? kXBytes : 0u));
        tma_load_3d(stage, &xmap, h * kD, n0, (int)b, &x_full[st.i]);
        tma_load_2d(stage + kXBytes, &pmap, 0, (int)(wk.bh * Np + n0), &x_full[st.i]);
        if (X3) tma_load_3d(stage + kDStage, &xrmap, h * kD, n0, (int)b, &x_full[st.i]);
      }
      // Drain: the newest load of each stage has landed before the CTA exits.
      for (int j = (i > ns ? i - ns : 0); j < i; j++)
        mbar_wait(&x_full[j % ns], (uint32_t)((j / ns) & 1), ab, nullptr, kWaitNs);
      mbar_wait(wz_full, 0, ab, nullptr, kWaitNs);
    }
  } else if (warp == 1) {
    // ------------------------------ logits issuer ------------------------------
    // Block q uses S buffer q % 3; it is rewritten only after the products of
    // block q - 3 (issued by the other warps) have completed.
    if (wk.ntiles > 0) {
      const uint32_t w0 = sdesc_lo(smem_u32(s_w), 16), we0 = w0 + (uint32_t)G * 4;
      const uint32_t wl0 = hilo ? w0 + (uint32_t)G * 6 : 0u, wl_step = hilo ? kGC * 4u : 0u;
      bool ok = mbar_wait_w(wz_full, 0, ab, status);
      Ring<kSBuf> sb;
      RingOf st(ns);
      int q = 0;
      for (int i = 0; ok && i < wk.ntiles; i++, st.next()) {
        if (!(ok = mbar_wait_w(&x_full[st.i], st.pass, ab, status))) break;
        const uint32_t xs = smem_u32(s_x + st.i * kDSt);
        const uint32_t x = sdesc_lo(xs, 16), xe = point_extra_lo(xs + kXBytes);
        const uint32_t xr = X3 ? sdesc_lo(xs + kDStage, 16) : 0u;
        uint32_t w = w0, we = we0, wl = wl0;
        for (int c = 0; c < nch; c++, q++, sb.next()) {
          if (q >= kSBuf && !(ok = mbar_wait_w(&pv_done[sb.i], sb.pass ^ 1u, ab, status))) break;
          tc_fence_after();
          issue_logits<true, kHiPx>(tmem + (uint32_t)sb.i * kGC, x, xe, w, we, wl, xr);
          mma_commit_w(&s_full[sb.i]);
          w += kGC * 4;
          we += kGC * 2;
          wl += wl_step;
        }
        mma_commit_w(&x_empty[st.i]);
      }
      mma_commit_w(&drain[0]);
      mbar_wait_w(&drain[0], 0, ab, nullptr, kWaitNs);
    }
  } else if (MODE == 3 && warp == 3) {
    // ------------------------------ P x [Z' | T2] issuer ------------------------------
    if (wk.ntiles > 0) {
      constexpr uint32_t idesc_pv = idesc_bf16(128, 2 * kD, false, false);
      const uint32_t z0 = sdesc_lo(smem_u32(s_z), 16);
      bool ok = mbar_wait_w(wz_full, 0, ab, status);
      Ring<kSBuf> sb;
      for (int i = 0; ok && i < wk.ntiles; i++) {
        if (i >= 1 && !(ok = mbar_wait_w(&o_free[0], (uint32_t)((i - 1) & 1), ab, status))) break;
        uint32_t z = z0;
        for (int c = 0; ok && c < nch; c++, sb.next()) {
#pragma unroll
          for (int j = 0; j < 2; j++, z += 512) {
            if (!(ok = mbar_wait_w(&p_ready[2 * sb.i + j], sb.pass, ab, status))) break;
            tc_fence_after();
            const uint32_t tP = tmem + (uint32_t)sb.i * kGC + (uint32_t)j * 64;
            const uint32_t tO = tmem + kO + (uint32_t)j * 2 * kD;
#pragma unroll
            for (int kk = 0; kk < 4; kk++) {
              const uint32_t hi = tP + da_col(kk), lo = hi + 16;
              mma_ts_w<kHi128>(tO, hi, z + kk * 2, idesc_pv, (c > 0 || kk > 0) ? 1u : 0u);
              mma_ts_w<kHi128>(tO, lo, z + kk * 2, idesc_pv, 1u);
              mma_ts_w<kHi128>(tO, hi, z + (uint32_t)G * 8 + kk * 2, idesc_pv, 1u);
            }
          }
          if (!ok) break;
          mma_commit_w(&pv_done[sb.i]);
        }
        mma_commit_w(&o_full[i % kOFull]);
      }
      mma_commit_w(&drain[1]);
      mbar_wait_w(&drain[1], 0, ab, nullptr, kWaitNs);
    }
  } else if (MODE != 3 && (warp == 2 || warp == 3)) {
    // ------------------------------ P x Z' issuers ------------------------------
    const int j = warp - 2;  // K-steps [4j, 4j + 4) of every block, accumulator O_j
    if (wk.ntiles > 0) {
      constexpr uint32_t idesc_pv = idesc_bf16(128, kD, false, false);
      // slots [64 j, 64 j + 64) of a block: 64-slot block 2 c + j of the Z' image
      const uint32_t z0 = sdesc_lo(smem_u32(s_z) + (uint32_t)j * 4096, 16);
      bool ok = mbar_wait_w(wz_full, 0, ab, status);
      Ring<kSBuf> sb;
      for (int i = 0; ok && i < wk.ntiles; i++) {
        const int ob = i & 1;
        const uint32_t tO = tmem + kO + (uint32_t)(j * 2 + ob) * kD;
        if (i >= 2 && !(ok = mbar_wait_w(&o_free[ob], (uint32_t)(((i >> 1) - 1) & 1), ab, status))) break;
        uint32_t z = z0;
        for (int c = 0; c < nch; c++, z += 512, sb.next()) {
          if (!(ok = mbar_wait_w(&p_ready[2 * sb.i + j], sb.pass, ab, status))) break;
          tc_fence_after();
          // weights of slots 64j.. (packed pairs; PS: at da_col(kk), lo pairs 16 on)
          const uint32_t tP = tmem + (uint32_t)sb.i * kGC + (uint32_t)j * (PS ? 64 : 32);
#pragma unroll
          for (int kk = 0; kk < 4; kk++) {
            const uint32_t tw = tP + (PS ? da_col(kk) : (uint32_t)kk * 8);
            mma_ts_w<kHi128>(tO, tw, z + kk * 2, idesc_pv, (c > 0 || kk > 0) ? 1u : 0u);
            if (PS) {
              mma_ts_w<kHi128>(tO, tw + 16, z + kk * 2, idesc_pv, 1u);
              mma_ts_w<kHi128>(tO, tw, z + (uint32_t)G * 4 + kk * 2, idesc_pv, 1u);
            }
          }
          mma_commit_w(&pv_done[sb.i]);
        }
        mma_commit_w(&o_full[i % kOFull]);
      }
      mma_commit_w(&drain[1 + j]);
      mbar_wait_w(&drain[1 + j], 0, ab, nullptr, kWaitNs);
    }
  } else if (warp >= kSoftmaxWarp0) {
    // ------------------------------ softmax warpgroups ------------------------------
    const int wg = (warp - kSoftmaxWarp0) >> 2;
    const int wq = warp & 3;  // TMEM sub-partition of this warp
    const int r = wq * 32 + lane + after_wait;
    const uint32_t lane_addr = (uint32_t)(wq * 32) << 16;
    bool ok = true;
    // Output of tile t: O_0 + O_1 (fixed order) -> bf16 -> global, 64 B per point.
    auto epilogue = [&](int t) -> bool {
      const int ob = (int)(t & 1);
      if (!mbar_wait(&o_full[t % kOFull], (uint32_t)((t / kOFull) & 1), ab, status)) return false;
      tc_fence_after();
      float R[kD];  // O_0 + O_1, in that order
      {
        uint32_t o0[32], o1[32];
        tmem_ld32(tmem + lane_addr + kO + (uint32_t)ob * kD, o0);
        tmem_ld32(tmem + lane_addr + kO + (uint32_t)(2 + ob) * kD, o1);
        tmem_wait_ld2(o0, o1);
#pragma unroll
        for (int k = 0; k < kD; k++) R[k] = __uint_as_float(o0[k]) + __uint_as_float(o1[k]);
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&o_free[ob]);
      const int64_t n = (wk.tile0 + t) * kTile + r;
      if (n < N) {
        const int64_t row = ((b * N + n) * H + h) * kD;
        if (X3) {
          // accumulate: a later slot range, added to the earlier ranges' output
          float4* dst = reinterpret_cast<float4*>(reinterpret_cast<float*>(out) + row);
#pragma unroll
          for (int k = 0; k < 8; k++) {
            const float4 p = accumulate ? dst[k] : make_float4(0.f, 0.f, 0.f, 0.f);
            dst[k] = make_float4(p.x + R[4 * k], p.y + R[4 * k + 1], p.z + R[4 * k + 2], p.w + R[4 * k + 3]);
          }
        } else if (MODE != 1) {
          uint4* dst = reinterpret_cast<uint4*>(out + row);
#pragma unroll
          for (int k = 0; k < 4; k++) {
            // MODE 2 over a later slot range: add the dfx of the earlier ranges
            uint4 p4 = make_uint4(0u, 0u, 0u, 0u);
            if (MODE == 2 && accumulate) p4 = dst[k];
            const uint32_t pw[4] = {p4.x, p4.y, p4.z, p4.w};
            uint32_t w[4];
#pragma unroll
            for (int e = 0; e < 4; e++)
              w[e] = pack_bf16(R[8 * k + 2 * e] + __uint_as_float(pw[e] << 16),
                               R[8 * k + 2 * e + 1] + __uint_as_float(pw[e] & 0xFFFF0000u));
            dst[k] = make_uint4(w[0], w[1], w[2], w[3]);
          }
        }
        if (MODE != 0) {
          // delta_n = v_n . R_n from the fp32 accumulators.
          const uint4* src = reinterpret_cast<const uint4*>(v + row);
          float acc = 0.f;
#pragma unroll
          for (int k = 0; k < 4; k++) {
            const uint4 q4 = src[k];
            const uint32_t w[4] = {q4.x, q4.y, q4.z, q4.w};
#pragma unroll
            for (int e = 0; e < 4; e++) {
              const int c0 = 8 * k + 2 * e;
              acc = fmaf(__uint_as_float(w[e] << 16), R[c0], acc);
              acc = fmaf(__uint_as_float(w[e] & 0xFFFF0000u), R[c0 + 1], acc);
            }
          }
          delta[wk.bh * N + n] = accumulate ? delta[wk.bh * N + n] + acc : acc;
        }
      }
      return true;
    };
    // MODE 3: delta_n = v_n . R2_n + v2_n . R_n and dfx_n = R2_n (R of z', R2 of t2).
    auto epilogue3 = [&](int t) -> bool {
      const int64_t n = (wk.tile0 + t) * kTile + r;
      const int64_t row = ((b * N + n) * H + h) * kD;
      uint4 va[4], vb[4];
      if (n < N) {
        const uint4* sa = reinterpret_cast<const uint4*>(v2 + row);
        const uint4* sb = reinterpret_cast<const uint4*>(v + row);
#pragma unroll
        for (int k = 0; k < 4; k++) va[k] = sa[k], vb[k] = sb[k];
      } else {
#pragma unroll
        for (int k = 0; k < 4; k++) va[k] = vb[k] = make_uint4(0u, 0u, 0u, 0u);
      }
      if (!mbar_wait(&o_full[t % kOFull], (uint32_t)((t / kOFull) & 1), ab, status)) return false;
      tc_fence_after();
      // Columns [col, col + 16) of the tile's accumulators, O_0 + O_1.
      auto load_sum = [&](uint32_t col, uint32_t (&o)[16]) {
        uint32_t o1[16];
        tmem_ld16(tmem + lane_addr + kO + col, o);
        tmem_ld16(tmem + lane_addr + kO + col + 2 * kD, o1);
        tmem_wait_ld(o);
        tmem_wait_ld(o1);
#pragma unroll
        for (int k = 0; k < 16; k++) o[k] = __float_as_uint(__uint_as_float(o[k]) + __uint_as_float(o1[k]));
      };
      uint32_t o[2][16];
      float da = 0.f, db = 0.f;
#pragma unroll
      for (int p = 0; p < 2; p++) {
        load_sum(16 * p, o[p]);
#pragma unroll
        for (int k = 0; k < 2; k++) {
          const uint4 q = va[2 * p + k];
          const uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
          for (int e = 0; e < 4; e++) {
            da = fmaf(__uint_as_float(w[e] << 16), __uint_as_float(o[p][8 * k + 2 * e]), da);
            da = fmaf(__uint_as_float(w[e] & 0xFFFF0000u), __uint_as_float(o[p][8 * k + 2 * e + 1]), da);
          }
        }
      }
      load_sum(kD, o[0]);
      load_sum(kD + 16, o[1]);
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&o_free[0]);
      if (n < N) {
        uint4* dst = reinterpret_cast<uint4*>(out + row);
#pragma unroll
        for (int k = 0; k < 4; k++) {
          const uint32_t wb[4] = {vb[k].x, vb[k].y, vb[k].z, vb[k].w};
          uint4 p4 = make_uint4(0u, 0u, 0u, 0u);
          if (accumulate) p4 = dst[k];
          const uint32_t pw[4] = {p4.x, p4.y, p4.z, p4.w};
          uint32_t w[4];
#pragma unroll
          for (int e = 0; e < 4; e++) {
            const int c0 = 8 * k + 2 * e;
            const float r0 = __uint_as_float(o[c0 >> 4][c0 & 15]), r1 = __uint_as_float(o[c0 >> 4][(c0 & 15) + 1]);
            w[e] = pack_bf16(r0 + __uint_as_float(pw[e] << 16), r1 + __uint_as_float(pw[e] & 0xFFFF0000u));
            db = fmaf(__uint_as_float(wb[e] << 16), r0, db);
            db = fmaf(__uint_as_float(wb[e] & 0xFFFF0000u), r1, db);
          }
          dst[k] = make_uint4(w[0], w[1], w[2], w[3]);
        }
        delta[wk.bh * N + n] = accumulate ? delta[wk.bh * N + n] + (db + da) : db + da;
      }
      return true;
    };
    // kDs: this warpgroup's sum_g w dS_g for point r of its current tile.
    float wds_acc = 0.f;
    int wds_tile = -1;
    auto flush_wds = [&]() {
      if (kDs && wds_tile >= 0) {
        const int64_t n = (wk.tile0 + wds_tile) * kTile + r;
        float* p = wds + ((int64_t)wg * gridDim.y + wk.bh) * N + n;
        if (n < N) *p = accumulate ? *p + wds_acc : wds_acc;
      }
      wds_acc = 0.f;
    };
    // Warpgroup wg takes the whole blocks q with q % kWGs == wg, so the warpgroups run
    // out of phase: one exponentiates while another waits.
    BlockPos pos(wg, nch);
    for (int q = wg; ok && q < total; q += kWGs, pos.step(kWGs, nch)) {
      const int i = pos.i, c = pos.c;
      const int bb = kWG3 ? wg : q % kSBuf;
      if (!(ok = mbar_wait(&s_full[bb], (uint32_t)((q / kSBuf) & 1), ab, status))) break;
      tc_fence_after();
      const uint32_t tS = tmem + lane_addr + (uint32_t)bb * kGC;
      if (kDs && i != wds_tile) {
        flush_wds();
        wds_tile = i;
      }
#pragma unroll
      for (int hf = 0; hf < 2; hf++) {
        const uint32_t tH = tS + (uint32_t)hf * 64;
        if constexpr (kDs)
          weights_hilo_half_ds(tH, s_ds + c * kGC + hf * 64, wds_acc);
        else if constexpr (PS)
          weights_hilo_half(tH);
        else
          weights_half(tH, tS + (uint32_t)hf * 32);
        tmem_wait_st();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&p_ready[2 * bb + hf]);
      }
      if constexpr (MODE == 3) {
        // A tile's output is drained by the warpgroup that took its last block, at once, as the
        // next tile's products wait for the accumulators.
        if (c == nch - 1 && !(ok = epilogue3(i))) break;
      } else {
        // The output of the previous tile is drained by the warpgroup that took the first
        // block of this tile, when the last products of that tile have long finished.
        if (c == 0 && i > 0 && !(ok = epilogue(i - 1))) break;
      }
    }
    if (MODE != 3 && ok && total > 0 && total % kWGs == wg) epilogue(wk.ntiles - 1);
    if (ok) flush_wds();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 1) tmem_dealloc(tmem, 512);
}

// =========================================================================================
// Statistics: lse_n = log sum_g exp(a_ng) (natural log) to lse[bh*N + n], and
// the point-extra row [1, 1, -lse2 in three bf16 parts, 0 x 3] (lse2 = lse*log2(e)) to
// px[bh*Np + n] (Np = N rounded up to a whole tile; padded points get -1e30 so
// that their weights vanish).
// nw softmax warpgroups (kStatsWGs, fewer where shared memory holds fewer x stages) take
// whole tiles (warpgroup w the tiles i with i % nw == w) and own S buffer w: a thread keeps its point's running (max, sum) over
// all slot blocks in registers and writes the point's results, so nothing is exchanged
// between warpgroups.  Warp 1 issues the logits of nw tiles in turn, block by block; an S
// buffer is rewritten once its second half is in registers, under the exponentials.
// MUFU and the softmax warps' issue slots bound it (a block's exponentials take 512 clocks
// and a loop of loads, maxima, exponentials and sums alone 640).  Warpgroups that shared
// tiles, each one half of every row, had to exchange their (max, sum) and waited on twice as
// many barriers per row (call at N = 262,144, H = 8: G = 1024 359 us, 256 118, 64 70; three
// warpgroups on whole tiles 349, 98, 56; four 330, 93, 54; four with a second issuing warp
// 356, 100, 56).
// smem: [W img G*96][x stages][constant extra][barriers]
// TMEM: S buffers [0, 128 kStatsWGs).
// =========================================================================================
// X3 (fp32 inputs): x arrives as bf16 hi and residual tiles (xmap, xrmap), one stage
// holding both, and the logits add x_r W'_hi.
constexpr int kStatsWGs = 4;
constexpr int kStatsThreads = 128 + 128 * kStatsWGs;
constexpr int kStatsMaxStages = 8;
template <bool split, bool X3>
__global__ void __launch_bounds__(kStatsThreads, 1)
    k_stats(const __grid_constant__ CUtensorMap xmap, const __grid_constant__ CUtensorMap xrmap,
            const uint8_t* __restrict__ wimg, float* __restrict__ lse, uint4* __restrict__ px, int64_t N,
            int64_t Np, int H, int G, int splits, int nst, int nw, uint32_t* status) {
  constexpr uint32_t kXSt = X3 ? 2 * kXBytes : kXBytes;  // x stage
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  // split (FS_DOT_BF16X2): the residual half of W' too (K = 80 logits).
  const uint32_t wbytes = (uint32_t)G * (split ? kWRow : 96);
  uint8_t* s_w = smem;
  uint8_t* s_x = s_w + wbytes;
  uint8_t* s_ex = s_x + (uint32_t)nst * kXSt;
  uint64_t* bars = reinterpret_cast<uint64_t*>(s_ex + kExBytes);
  uint64_t* w_full = bars;
  uint64_t* x_full = bars + 1;
  uint64_t* x_empty = x_full + kStatsMaxStages;
  uint64_t* s_full = x_empty + kStatsMaxStages;
  uint64_t* s_free = s_full + kStatsWGs;
  uint64_t* drain = s_free + kStatsWGs;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain + 1);
  Abort* ab = reinterpret_cast<Abort*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const Work wk = work_of(N, splits, blockIdx.x, blockIdx.y);
  const int64_t b = wk.bh / H;
  const int h = (int)(wk.bh % H);
  const int nch = G / kGC;

  if (threadIdx.x == 0) {
    mbar_init(w_full, 1);
    for (int s = 0; s < nst; s++) {
      mbar_init(&x_full[s], 1);
      mbar_init(&x_empty[s], 1);
    }
    for (int i = 0; i < kStatsWGs; i++) {
      mbar_init(&s_full[i], 1);
      mbar_init(&s_free[i], 4);
    }
    mbar_init(drain, 1);
    ab->flag = 0;
    fence_mbar_init();
  }
  write_const_extra(s_ex);
  fence_proxy_async_smem();
  if (warp == 1) tmem_alloc(tmem_slot, 512);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  grid_trigger();
  grid_wait(wimg);

  if (warp == 0) {
    if (lane == 0 && wk.ntiles > 0) {
      prefetch_tmap(&xmap);
      if (X3) prefetch_tmap(&xrmap);
      mbar_expect_tx(w_full, wbytes);
      load_images(s_w, wimg + (size_t)h * G * kWRow, wbytes, w_full);
      int i = 0, s = 0;
      uint32_t pass = 0;
      for (; i < wk.ntiles; i++) {
        if (i >= nst && !mbar_wait(&x_empty[s], pass ^ 1u, ab, status)) break;
        const int n0 = (int)((wk.tile0 + i) * kTile);
        mbar_expect_tx(&x_full[s], kXSt);
        tma_load_3d(s_x + s * kXSt, &xmap, h * kD, n0, (int)b, &x_full[s]);
        if (X3) tma_load_3d(s_x + s * kXSt + kXBytes, &xrmap, h * kD, n0, (int)b, &x_full[s]);
        if (++s == nst) s = 0, pass ^= 1u;
      }
      for (int j = (i > nst ? i - nst : 0); j < i; j++)
        mbar_wait(&x_full[j % nst], (uint32_t)((j / nst) & 1), ab, nullptr, kWaitNs);
      mbar_wait(w_full, 0, ab, nullptr, kWaitNs);
    }
  } else if (warp == 1) {
    if (wk.ntiles > 0) {
      const uint32_t w0 = sdesc_lo(smem_u32(s_w), 16), we0 = w0 + (uint32_t)G * 4;
      const uint32_t wl0 = split ? w0 + (uint32_t)G * 6 : 0u, xe = const_extra_lo(smem_u32(s_ex));
      bool ok = mbar_wait_w(w_full, 0, ab, status);
      uint32_t par = 1;  // parity of the S buffers' previous release
      int s0 = 0;        // stage of the first of the tiles taken together
      uint32_t pass0 = 0;
      for (int i0 = 0; ok && i0 < wk.ntiles; i0 += nw) {
        const int nt = min(nw, wk.ntiles - i0);
        for (int c = 0; ok && c < nch; c++, par ^= 1u) {
          const uint32_t w = w0 + (uint32_t)c * (kGC * 4), we = we0 + (uint32_t)c * (kGC * 2);
          const uint32_t wl = split ? wl0 + (uint32_t)c * (kGC * 4) : 0u;
          int s = s0;
          uint32_t pass = pass0;
          for (int k = 0; k < nt; k++) {
            if (c == 0 && !(ok = mbar_wait_w(&x_full[s], pass, ab, status))) break;
            if (i0 + c > 0 && !(ok = mbar_wait_w(&s_free[k], par, ab, status))) break;
            tc_fence_after();
            const uint32_t xs = smem_u32(s_x + s * kXSt);
            issue_logits<true, kHi32>(tmem + (uint32_t)k * kGC, sdesc_lo(xs, 16), xe, w, we, wl,
                                      X3 ? sdesc_lo(xs + kXBytes, 16) : 0u);
            mma_commit_w(&s_full[k]);
            if (c == nch - 1) mma_commit_w(&x_empty[s]);
            if (++s == nst) s = 0, pass ^= 1u;
          }
        }
        s0 += nt;
        if (s0 >= nst) s0 -= nst, pass0 ^= 1u;
      }
      mma_commit_w(drain);
      mbar_wait_w(drain, 0, ab, nullptr, kWaitNs);
    }
  } else if (warp >= kSoftmaxWarp0) {
    const int wg = (warp - kSoftmaxWarp0) >> 2;
    const int wq = warp & 3;
    const int r = wq * 32 + lane;
    const uint32_t tS = tmem + ((uint32_t)(wq * 32) << 16) + (uint32_t)wg * kGC;
    bool ok = true;
    uint32_t par = 0;
    for (int i = wg; ok && wg < nw && i < wk.ntiles; i += nw) {
      float m = -INFINITY, l = 0.f;
      for (int c = 0; c < nch; c++, par ^= 1u) {
        if (!(ok = mbar_wait(&s_full[wg], par, ab, status))) break;
        tc_fence_after();
#pragma unroll 1
        for (int hf = 0; hf < 2; hf++) {
          uint32_t v[2][32];
          tmem_ld32(tS + 64 * hf, v[0]);
          tmem_ld32(tS + 64 * hf + 32, v[1]);
          tmem_wait_ld2(v[0], v[1]);
          if (hf == 1) {
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&s_free[wg]);
          }
          float t[22];
#pragma unroll
          for (int k = 0; k < 21; k++)
            t[k] = max3(__uint_as_float(v[(3 * k) >> 5][(3 * k) & 31]),
                        __uint_as_float(v[(3 * k + 1) >> 5][(3 * k + 1) & 31]),
                        __uint_as_float(v[(3 * k + 2) >> 5][(3 * k + 2) & 31]));
          t[21] = fmaxf(__uint_as_float(v[1][31]), m);
#pragma unroll
          for (int k = 0; k < 7; k++) t[k] = max3(t[3 * k], t[3 * k + 1], t[3 * k + 2]);
          const float mn = max3(max3(t[0], t[1], t[2]), max3(t[3], t[4], t[5]), fmaxf(t[6], t[21]));
          const uint32_t nmb = __float_as_uint(-mn);
          const uint64_t nm2 = pack2(nmb, nmb);
#pragma unroll
          for (int j = 0; j < 2; j++)
#pragma unroll
            for (int k = 0; k < 16; k++) {
              const uint64_t a = add2(pack2(v[j][2 * k], v[j][2 * k + 1]), nm2);
              v[j][2 * k] = __float_as_uint(ex2(lo_f(a)));
              v[j][2 * k + 1] = __float_as_uint(ex2(hi_f(a)));
            }
          uint64_t acc[16];
#pragma unroll
          for (int k = 0; k < 16; k++)
            acc[k] = add2(pack2(v[0][2 * k], v[0][2 * k + 1]), pack2(v[1][2 * k], v[1][2 * k + 1]));
#pragma unroll
          for (int w = 8; w >= 1; w >>= 1)
#pragma unroll
            for (int k = 0; k < w; k++) acc[k] = add2(acc[k], acc[k + w]);
          l = l * ex2(m - mn) + (lo_f(acc[0]) + hi_f(acc[0]));
          m = mn;
        }
      }
      if (!ok) break;
      const int64_t n = (wk.tile0 + i) * kTile + r;
      const float lse2 = m + log2f(l);
      if (n < Np) {
        px[wk.bh * Np + n] = extra_row3(n < N ? -lse2 : -1e30f);
        if (n < N) lse[wk.bh * N + n] = lse2 * kLn2;
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 1) tmem_dealloc(tmem, 512);
}

// =========================================================================================
// Slice (slot-owned, split over points), slot-major: CTA (p, bh, j) owns the
// 128-slot block j of head h and point split p and computes for its slots
//   U_g = sum_n w_ng f_n,  S_g = sum_n w_ng,  w_ng = 2^(a2_ng - lse2_n).
// The logits are formed transposed (M = 128 slots, N = 128 points), so TMEM
// lane = slot and column = point; the point-extra rows of the tile arrive by
// TMA with it, so the accumulator holds log2 of the weights.  The bf16 weights
// written back in place serve directly as the TMEM A operand of
// U|S += E [F | 1] (K = points), so the weight tile never passes through
// shared memory.
// Writes part[p][bh][g][0..32] = (U_g, S_g).
// smem: [W img block 128*96][stages: x | F_lo F_hi ones | point extra (2 halves)][barriers]
// TMEM: S buffers [0, 384); U|S accumulators A_0 [384, 432), A_1 [432, 480).
// Warp 1 issues the logits of every tile; softmax warpgroup wg takes the whole
// tiles i with i % 2 == wg, and warp 2 + wg issues their products into its own
// accumulator A_wg (the two are summed in a fixed order).
// =========================================================================================
constexpr uint32_t kStageBytes = kXBytes + 3 * kFBlock + 2 * kPxBytes;  // x, [F | 1], point extra
constexpr uint32_t kWBlock = 128 * kWRow;                               // one 128-slot block of the W image

// Flushes.  The tensor cores' fp32 accumulation over a CTA's long point range (a
// thousand and more K steps into one accumulator) loses ~2^-25 of the running sum per
// step, always towards zero: at 27,600 points 4e-5 relative, and the temperature
// gradient magnifies errors of the token gradients many times over (its sum over
// (n, g) cancels to ~1e-5 of its terms' magnitude).  So each accumulator's chain is
// restarted every kSliceFlush of its issuer's tiles, after its warpgroup has added
// what it holds into fp32 registers (round to nearest).  With single bf16 products the
// weights' own rounding (~3e-3 relative in the tokens) dwarfs the drift (~1e-4 at 55,000
// points per CTA), and the waits on a chain flushed every 4 tiles cost the plain slice 4%:
// there a chain of 64 tiles (512 K steps) keeps the drift at the level of a short CTA's
// however long the CTA's range is, at no measurable cost.
template <bool split>
__device__ __forceinline__ bool slice_flush_at(int i) { return ((i >> 1) % (split ? 4 : 64)) == 0; }

// X3 (fp32 inputs): each stage also holds the residual tiles of x and fx (xrmap,
// frmap); the logits add x_r W'_hi and the products add P_hi F_r (N = 32: U only).
// Its stages are larger, so there are half as many.
template <bool split, bool X3>
__global__ void __launch_bounds__(kThreads, 1)
    k_slice(const __grid_constant__ CUtensorMap xmap, const __grid_constant__ CUtensorMap fmap,
            const __grid_constant__ CUtensorMap pmap, const __grid_constant__ CUtensorMap xrmap,
            const __grid_constant__ CUtensorMap frmap, const uint8_t* __restrict__ wimg, float* __restrict__ part,
            int64_t N, int64_t Np, int H, int G, int splits, uint32_t* status) {
  constexpr int kSBuft = X3 ? kSliceStages / 2 : kSliceStages;
  constexpr uint32_t kStB = kStageBytes + (X3 ? kXBytes + 2 * kFBlock : 0u);
  constexpr uint32_t kXROff = kStageBytes, kFROff = kStageBytes + kXBytes;
  // split (FS_DOT_BF16X2): logits with both halves of W' (K = 80), and the
  // weights as hi + lo bf16 halves in the products (twice the product MMAs).
  // Grid (slot block, point split, bh): the CTAs of all slot blocks of one point
  // range are adjacent in launch order, run together and share each x / F tile
  // through L2 instead of re-reading it from DRAM once per slot block.
  const int g_base = blockIdx.x * kGC;
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* s_w = smem;
  uint8_t* s_st = s_w + kWBlock;
  uint64_t* bars = reinterpret_cast<uint64_t*>(s_st + kSBuft * kStB);
  uint64_t* w_full = bars;
  uint64_t* x_full = bars + 1;
  uint64_t* st_empty = x_full + kSBuft;
  uint64_t* s_full = st_empty + kSBuft;
  uint64_t* p_ready = s_full + kSBuf;   // [S buffer][half]
  uint64_t* pv_done = p_ready + 2 * kSBuf;
  uint64_t* acc_full = pv_done + kSBuf;
  uint64_t* acc_done = acc_full + 1;  // [issuer][its tiles' parity]: a tile's products complete
  uint64_t* wt_ready = acc_done + 4;  // single-level products: the W' image is in TMEM
  uint64_t* drain = wt_ready + 1;  // one per issuing warp
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain + 3);
  Abort* ab = reinterpret_cast<Abort*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const Work wk = work_of(N, splits, blockIdx.y, blockIdx.z);
  const int64_t b = wk.bh / H;
  const int h = (int)(wk.bh % H);
  constexpr uint32_t kA = kSBuf * kGC;  // TMEM column base of the accumulators
  constexpr uint32_t kFOff = kXBytes, kPOff = kXBytes + 3 * kFBlock;
  // With single-level products the slot block's W' image (W' and its extra block: 24
  // columns) fits in the 32 TMEM columns after the accumulators, and the logits read
  // only their point side from shared memory.
  constexpr bool kWT = !split && !X3;
  constexpr uint32_t kTW = kA + 96;

  if (threadIdx.x == 0) {
    mbar_init(w_full, 1);
    for (int s = 0; s < kSBuft; s++) {
      mbar_init(&x_full[s], 1);
      mbar_init(&st_empty[s], 2);  // the logits issuer and the tile's product issuer
    }
    for (int i = 0; i < kSBuf; i++) {
      mbar_init(&s_full[i], 1);
      mbar_init(&p_ready[i], 4);  // the four warps of the warpgroup that took the tile
      mbar_init(&p_ready[kSBuf + i], 4);
      mbar_init(&pv_done[i], 1);
    }
    mbar_init(acc_full, 2);
    for (int i = 0; i < 4; i++) mbar_init(&acc_done[i], 1);
    mbar_init(wt_ready, 4);
    for (int i = 0; i < 3; i++) mbar_init(&drain[i], 1);
    ab->flag = 0;
    fence_mbar_init();
  }
  for (int s = 0; s < kSBuft; s++) zero_smem(s_st + s * kStB + kPOff + kPxBytes, kPxBytes);
  // Constant "ones" block of every stage: row n = [1, 0 x 15] (32B swizzle).
  for (int idx = threadIdx.x; idx < kSBuft * kTile; idx += kThreads) {
    const int s = idx / kTile, r = idx % kTile;
    const uint32_t base = smem_u32(s_st + s * kStB + kFOff + 2 * kFBlock) +
                          (uint32_t)((r >> 3) * 256 + (r & 7) * 32);
    const uint32_t sw = (uint32_t)((r & 7) >> 2);
    st_shared_v4(base + ((0u ^ sw) << 4), 0x3F80u, 0u, 0u, 0u);
    st_shared_v4(base + ((1u ^ sw) << 4), 0u, 0u, 0u, 0u);
  }
  fence_proxy_async_smem();
  if (warp == 1) tmem_alloc(tmem_slot, 512);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  grid_trigger();
  grid_wait(wimg);

  if (warp == 0) {
    if (lane == 0) {
      prefetch_tmap(&xmap);
      prefetch_tmap(&fmap);
      prefetch_tmap(&pmap);
      if (X3) {
        prefetch_tmap(&xrmap);
        prefetch_tmap(&frmap);
      }
      // The slot block's rows of the W image: 128 rows of W' (64 B) then 128 rows of
      // the extra block (32 B); the global image holds G rows of each.
      mbar_expect_tx(w_full, split ? kWBlock : kGC * 96);
      const uint8_t* src = wimg + (size_t)h * G * kWRow;
      load_images(s_w, src + (size_t)g_base * 64, kGC * 64, w_full);
      load_images(s_w + kGC * 64, src + (size_t)G * 64 + (size_t)g_base * 32, kGC * 32, w_full);
      if (split) load_images(s_w + kGC * 96, src + (size_t)G * 96 + (size_t)g_base * 64, kGC * 64, w_full);
      int i = 0;
      for (; i < wk.ntiles; i++) {
        const int s = i % kSBuft;
        if (i >= kSBuft &&
            !mbar_wait(&st_empty[s], (uint32_t)(((i / kSBuft) - 1) & 1), ab, status))
          break;
        uint8_t* st = s_st + s * kStB;
        const int n0 = (int)((wk.tile0 + i) * kTile);
        mbar_expect_tx(&x_full[s], kXBytes + 2 * kFBlock + kPxBytes + (X3 ? kXBytes + 2 * kFBlock : 0u));
        tma_load_3d(st, &xmap, h * kD, n0, (int)b, &x_full[s]);
        tma_load_3d(st + kFOff, &fmap, h * kD, n0, (int)b, &x_full[s]);
        tma_load_3d(st + kFOff + kFBlock, &fmap, h * kD + 16, n0, (int)b, &x_full[s]);
        tma_load_2d(st + kPOff, &pmap, 0, (int)(wk.bh * Np + n0), &x_full[s]);
        if (X3) {
          tma_load_3d(st + kXROff, &xrmap, h * kD, n0, (int)b, &x_full[s]);
          tma_load_3d(st + kFROff, &frmap, h * kD, n0, (int)b, &x_full[s]);
          tma_load_3d(st + kFROff + kFBlock, &frmap, h * kD + 16, n0, (int)b, &x_full[s]);
        }
      }
      for (int j = (i > kSBuft ? i - kSBuft : 0); j < i; j++)
        mbar_wait(&x_full[j % kSBuft], (uint32_t)((j / kSBuft) & 1), ab, nullptr, kWaitNs);
      mbar_wait(w_full, 0, ab, nullptr, kWaitNs);
    }
  } else if (warp == 1) {
    // ------------------------------ logits issuer (transposed) ------------------------------
    {
      const uint32_t w = sdesc_lo(smem_u32(s_w), 16), we = w + kGC * 4;
      bool ok = mbar_wait_w(w_full, 0, ab, status);
      if (kWT && ok) {
        ok = mbar_wait_w(wt_ready, 0, ab, status);
        tc_fence_after();
      }
      Ring<kSBuft> st;
      Ring<kSBuf> sb;
      for (int i = 0; ok && i < wk.ntiles; i++, st.next(), sb.next()) {
        if (!(ok = mbar_wait_w(&x_full[st.i], st.pass, ab, status))) break;
        if (i >= kSBuf && !(ok = mbar_wait_w(&pv_done[sb.i], sb.pass ^ 1u, ab, status))) break;
        tc_fence_after();
        const uint32_t xs = smem_u32(s_st + st.i * kStB);
        const uint32_t x = sdesc_lo(xs, 16), xe = point_extra_lo(xs + kPOff);
        const uint32_t tD = tmem + (uint32_t)sb.i * kGC;
        if (kWT) {
          constexpr uint32_t idesc = idesc_bf16(128, kGC, false, false);
          mma_ts_w<kHi64>(tD, tmem + kTW, x, idesc, 0u);
          mma_ts_w<kHi64>(tD, tmem + kTW + 8, x + 2, idesc, 1u);
          mma_ts_w<kHiPx>(tD, tmem + kTW + 16, xe, idesc, 1u);
        } else {
          issue_logits<false, kHiPx>(tD, x, xe, w, we, split ? w + kGC * 6 : 0u, X3 ? sdesc_lo(xs + kXROff, 16) : 0u);
        }
        mma_commit_w(&s_full[sb.i]);
        mma_commit_w(&st_empty[st.i]);
      }
      mma_commit_w(&drain[0]);
      mbar_wait_w(&drain[0], 0, ab, nullptr, kWaitNs);
    }
  } else if (warp == 2 || warp == 3) {
    // ------------------------------ product issuers ------------------------------
    const int j = warp - 2;  // tiles i with i % 2 == j, accumulator A_j
    {
      constexpr uint32_t idesc_sl = idesc_bf16(128, 48, false, true);
      bool ok = true;
      Ring<kSBuft> st;
      Ring<kSBuf> sb;
      if (j == 1) st.next(), sb.next();
      for (int i = j; ok && i < wk.ntiles; i += 2) {
        const uint32_t tE = tmem + (uint32_t)sb.i * kGC;  // packed weights of the 128 points
        const uint32_t f = sdesc_lo(smem_u32(s_st + st.i * kStB) + kFOff, kFBlock);
        const uint32_t fr = f - kFOff / 16 + kFROff / 16;
        const uint32_t tacc = tmem + kA + (uint32_t)j * 48;
        // A chain restarts at this issuer's first tile and at every flush tile (its
        // warpgroup has moved the earlier tiles' sums to registers by then).
        const bool fresh = i < 2 || slice_flush_at<split>(i);
#pragma unroll
        for (int kk = 0; kk < 8; kk++) {
          if ((kk & 3) == 0) {  // a half's weights
            if (!(ok = mbar_wait_w(&p_ready[2 * sb.i + (kk >> 2)], sb.pass, ab, status))) break;
            tc_fence_after();
          }
          // 16 points' packed weights: columns kk * 8, or with split products at da_col(kk)
          const uint32_t tw = tE + (split ? da_col(kk) : (uint32_t)kk * 8);
          mma_ts_w<kHi32>(tacc, tw, f + kk * 32, idesc_sl, (!fresh || kk > 0) ? 1u : 0u);
          // The residual halves of the weights: U and S to ~2^-16.
          if (split) mma_ts_w<kHi32>(tacc, tw + 16, f + kk * 32, idesc_sl, 1u);
          if (X3)  // the weights against fx's residual half (U only)
            mma_ts_w<kHi32>(tacc, tw, fr + kk * 32, idesc_bf16(128, 32, false, true), 1u);
        }
        mma_commit_w(&pv_done[sb.i]);
        mma_commit_w(&st_empty[st.i]);
        mma_commit_w(&acc_done[acc_done_of(i)]);
        st.next(), st.next();
        sb.next(), sb.next();
      }
      if (ok) mma_commit_w(acc_full);
      mma_commit_w(&drain[1 + j]);
      mbar_wait_w(&drain[1 + j], 0, ab, nullptr, kWaitNs);
    }
  } else if (warp >= kSoftmaxWarp0) {
    const int wg = (warp - kSoftmaxWarp0) >> 2;
    const int wq = warp & 3;
    const int r = wq * 32 + lane;  // TMEM lane: slot g_base + r
    const uint32_t lane_addr = (uint32_t)(wq * 32) << 16;
    bool ok = true;
    if (kWT && wg == 0) {
      // Slot r's W' row (64B-swizzled) and extra row (32B-swizzled) from the block's image
      // in shared memory into TMEM columns [kTW, kTW + 24) of lane r (packed bf16 pairs).
      if ((ok = mbar_wait(w_full, 0, ab, status))) {
        uint32_t hi[16], ex[16];
#pragma unroll
        for (int c = 0; c < 16; c++) {
          hi[c] = *reinterpret_cast<const uint32_t*>(s_w + off_sw64(r, 2 * c));
          ex[c] = c < 8 ? *reinterpret_cast<const uint32_t*>(s_w + kGC * 64 + off_sw32(r, 2 * c)) : 0u;
        }
        tmem_st16(tmem + lane_addr + kTW, hi);
        tmem_st16(tmem + lane_addr + kTW + 16, ex);
        tmem_wait_st();
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(wt_ready);
    }
    // This warpgroup's share of (U, S) for slot r, moved out of A_wg at every flush.
    float acc[kD + 1];
#pragma unroll
    for (int k = 0; k <= kD; k++) acc[k] = 0.f;
    const uint32_t tA = tmem + lane_addr + kA + (uint32_t)wg * 48;
    auto add_acc = [&]() {
      uint32_t u[32], sv[16];
      tmem_ld32(tA, u);
      tmem_ld16(tA + 32, sv);
      tmem_wait_ld(u, sv);
#pragma unroll
      for (int k = 0; k < kD; k++) acc[k] += __uint_as_float(u[k]);
      acc[kD] += __uint_as_float(sv[0]);
    };
    // Warpgroup wg takes the whole tiles i with i % 2 == wg (out of phase with the other).
    for (int i = wg; ok && i < wk.ntiles; i += 2) {
      const int bb = i % kSBuf;
      if (!(ok = mbar_wait(&s_full[bb], (uint32_t)((i / kSBuf) & 1), ab, status))) break;
      tc_fence_after();
      const uint32_t tS = tmem + lane_addr + (uint32_t)bb * kGC;
#pragma unroll
      for (int hf = 0; hf < 2; hf++) {
        if constexpr (split)
          weights_hilo_half(tS + (uint32_t)hf * 64);
        else
          weights_half(tS + (uint32_t)hf * 64, tS + (uint32_t)hf * 32);
        tmem_wait_st();
        if (hf == 0 && i >= 2 && slice_flush_at<split>(i)) {
          // The products of this warpgroup's tiles up to i - 2 are complete.
          if (!(ok = mbar_wait(&acc_done[acc_done_of(i - 2)], acc_done_phase(i - 2), ab, status))) break;
          tc_fence_after();
          add_acc();
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&p_ready[2 * bb + hf]);
      }
    }
    const int64_t BH = gridDim.z;
    const bool have = ok && wk.ntiles > 0 && mbar_wait(acc_full, 0, ab, status);
    // What the accumulators hold since the last flush, then the two warpgroups' shares added
    // in a fixed order.  The 128 rows of the partials are contiguous: gathered in the stages'
    // memory (every load has landed and been read) they leave as one bulk copy.  (Stored by
    // their threads, 132 bytes apart, and the shares added through global memory, split slice
    // call at N = 32,768, H = 8, G = 64: 27.3 us against 21.)
    if (have && wg < wk.ntiles) {
      tc_fence_after();
      add_acc();
    }
    float* s_out = reinterpret_cast<float*>(s_st);
    float* row = s_out + r * (kD + 1);
    if (wg == 1)
      for (int k = 0; k <= kD; k++) row[k] = acc[k];
    named_barrier(1, 256);
    if (wg == 0) {
      for (int k = 0; k <= kD; k++) row[k] = acc[k] + row[k];
      fence_proxy_async_smem();
      named_barrier(2, 128);
      if (r == 0)
        bulk_store(part + (((int64_t)blockIdx.y * BH + wk.bh) * G + g_base) * (kD + 1), s_out, kGC * (kD + 1) * 4);
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 1) tmem_dealloc(tmem, 512);
}

// One slice CTA per (point split, batch-head, 128-slot block).
int slice_blocks(const Shape& s) { return s.G / kGC < 1 ? 1 : s.G / kGC; }
int slice_splits(const Shape& s) { return point_splits(s, (int)(s.BH() * slice_blocks(s)), 1); }

// fp32 point tensors take the tensor-core path with every operand as two bf16 halves
// (x, fx and W', the weights, z'): the X3 kernels.  Their inputs are first split
// into bf16 hi and residual tensors in the workspace (k_prep).
bool x3_shape(const Shape& s) { return s.dtype == FS_F32; }

// The X3 deslice holds both halves of W' and of z' in shared memory, which fits up to
// 512 slots; past that it runs over ranges of `size` slots (a multiple of 128), each
// with the full lse, adding its output to the earlier ranges': as few as fit (a range
// re-reads x), of equal size but for the last.
constexpr int kX3SlotsMax = 512;
struct X3Ranges {
  int n, size;
};
X3Ranges x3_ranges(const Shape& s0) {
  const int Gp = (s0.G + kGC - 1) / kGC * kGC;
  if (s0.dtype != FS_F32 || s0.G <= kX3SlotsMax) return {1, Gp};
  const int n = (Gp + kX3SlotsMax - 1) / kX3SlotsMax;
  return {n, (Gp / kGC + n - 1) / n * kGC};
}
size_t half_bytes(const Shape& s) { return align_up((size_t)s.B * s.N * s.H * s.d * 2, 256); }

size_t smem_deslice(int G, bool hilo, int mode = 0, bool ps = false, bool x3 = false) {
  return 1024 + (size_t)G * ((hilo ? kWRow : 96) + (mode == 3 ? 256 : ps ? 128 : 64)) +
         (mode >= 2 ? align_up((size_t)G * 4, 1024) : 0) +
         (mode == 3 ? 1 : kStages) * (kDStage + (x3 ? kXBytes : 0)) + 512;
}
// Shared memory of the statistics pass and, from what W' leaves, its x stages.
size_t smem_stats(int G, bool split, bool x3, int nst) {
  return 1024 + (size_t)G * (split ? kWRow : 96) + (size_t)nst * kXBytes * (x3 ? 2 : 1) + kExBytes + 512;
}
size_t smem_slice(bool x3 = false) {
  return 1024 + (size_t)kWBlock +
         (x3 ? (size_t)(kSliceStages / 2) * (kStageBytes + kXBytes + 2 * kFBlock) : (size_t)kSliceStages * kStageBytes) +
         512;
}

// Statistics into lse [B,H,N] and the point-extra rows at px.  xr: x's residual
// half (X3), else null.
cudaError_t run_stats(const Shape& s, const void* x, const void* xr, const uint8_t* wimg, float* lse, void* px,
                      uint32_t* status, cudaStream_t st) {
  CUtensorMap xmap, xrmap;
  if (!make_point_map(&xmap, x, s, kD, CU_TENSOR_MAP_SWIZZLE_64B)) return cudaErrorInvalidValue;
  if (!make_point_map(&xrmap, xr ? xr : x, s, kD, CU_TENSOR_MAP_SWIZZLE_64B)) return cudaErrorInvalidValue;
  const int P = point_splits(s, (int)s.BH(), s.G / kGC);
  const bool x3 = xr != nullptr;
  const bool split = s.dot == FS_DOT_BF16X2 || x3;
  int nst = kStatsMaxStages;
  while (nst > 1 && smem_stats(s.G, split, x3, nst) > kMaxSmem) nst--;
  const size_t sm = smem_stats(s.G, split, x3, nst);
  const auto kernel = x3 ? k_stats<true, true> : (split ? k_stats<true, false> : k_stats<false, false>);
  cudaError_t e = set_smem(kernel, sm);
  if (e != cudaSuccess) return e;
  return launch(kernel, dim3((unsigned)P, (unsigned)s.BH()), dim3(kStatsThreads), sm, st, xmap, xrmap, wimg, lse,
                static_cast<uint4*>(px), s.N, padded_n(s), s.H, s.G, P, nst, std::min(nst, kStatsWGs), status);
}

}  // namespace

// The slice on prepared operands (defined below, after the C-ABI-facing helpers).
cudaError_t run_slice(const Shape& s, int G, const void* x, const void* f, const void* xr, const void* fr,
                      const uint8_t* wimg, void* px, float* tokens, float* wsum, int finalize, float* part,
                      uint32_t* status, cudaStream_t st);

bool tc_forward_supported(const Shape& s) {
  // TMA coordinates and the kernels' block counters are 32-bit.
  const int64_t np = (s.N + kTile - 1) / kTile * kTile;
  // fp32 inputs take the tensor cores only when there is enough work to pay for
  // splitting their inputs: B*N*H*G >= 2^24 (smaller problems keep the exact fp32
  // SIMT kernels).  Their deslice runs over slot ranges past 512 slots (X3 ranges).
  const bool fp32_ok = s.dtype == FS_F32 && (double)s.BH() * s.N * s.G >= 16777216.0;
  return (s.dtype == FS_BF16 || fp32_ok) && s.d == kD && s.G <= 1024 && s.N >= 1 &&
         s.BH() * np < (int64_t(1) << 31) && encode_fn() != nullptr;
}

int tc_stats_launch_count(const Shape& s) { return 2 /*prep, stats*/; }

int tc_forward_launch_count(const Shape& s) {
  return 4 /*prep, stats, slice, reduce*/ + 1 /*prep*/ + x3_ranges(s).n /*deslice*/;
}

size_t tc_slice_partials_bytes(const Shape& s0) {
  if (!tc_forward_supported(s0)) return 0;
  const Shape s = tc_padded(s0);
  // (sized for the most splits that a size can take, so that a shape's scratch, and with it
  // what fits a fixed one, does not hang on the choice of splits)
  return (size_t)wave_splits(s, (int)(s.BH() * slice_blocks(s))) * s.BH() * s.G * (kD + 1) * sizeof(float);
}
// Layouts of the prepared operands: slice [W img | px | (X3) x hi, x r, fx hi, fx r];
// deslice and statistics [W img | Z' img | px | (X3) x hi, x r].
size_t tc_slice_prep_bytes(const Shape& s0) {
  const Shape s = tc_padded(s0);
  return tc_forward_supported(s0)
             ? align_up(w_image_bytes(s), 256) + align_up(px_bytes(s), 256) + (x3_shape(s) ? 4 * half_bytes(s) : 0)
             : 0;
}
size_t tc_deslice_prep_bytes(const Shape& s0) {
  const Shape s = tc_padded(s0);
  return tc_forward_supported(s0) ? align_up(w_image_bytes(s), 256) + align_up(z_image_bytes(s), 256) +
                                        align_up(px_bytes(s), 256) + (x3_shape(s) ? 2 * half_bytes(s) : 0)
                                  : 0;
}

cudaError_t tc_stats(const Shape& s0, const void* x, const float* W, const float* bias, const float* tau, float* lse,
                     void* prep, bool reset, uint32_t* status, cudaStream_t st) {
  const Shape s = tc_padded(s0);
  uint8_t* wimg = static_cast<uint8_t*>(prep);
  uint8_t* px = wimg + align_up(w_image_bytes(s), 256) + align_up(z_image_bytes(s), 256);
  uint8_t* xh = px + align_up(px_bytes(s), 256);
  const bool x3 = x3_shape(s);
  Prepare p(s, s0.G, tau, status, reset);
  p.weights(W, bias, wimg);
  if (x3) p.split(s, x, xh, half_bytes(s));
  if (cudaError_t e = p.run(st)) return e;
  return run_stats(s, x3 ? xh : x, x3 ? xh + half_bytes(s) : nullptr, wimg, lse, px, status, st);
}

// The slice with its statistics pass (lse an output) or, with given, without it.
static cudaError_t slice_with_prep(const Shape& s0, const void* x, const void* f, const float* W, const float* bias,
                                   const float* tau, float* tokens, float* wsum, float* lse, const float* given,
                                   int finalize, float* part, void* prep, bool reset, uint32_t* status,
                                   cudaStream_t st) {
  const Shape s = tc_padded(s0);
  uint8_t* wimg = static_cast<uint8_t*>(prep);
  uint8_t* px = wimg + align_up(w_image_bytes(s), 256);
  uint8_t* xh = px + align_up(px_bytes(s), 256);
  uint8_t* fh = xh + 2 * half_bytes(s);
  Prepare p(s, s0.G, tau, status, reset);
  p.weights(W, bias, wimg);
  if (given) p.rows(given, px);
  const void *xr = nullptr, *fr = nullptr;
  if (x3_shape(s)) {
    p.split(s, x, xh, half_bytes(s));
    p.split(s, f, fh, half_bytes(s));
    x = xh, xr = xh + half_bytes(s);
    f = fh, fr = fh + half_bytes(s);
  }
  cudaError_t e = p.run(st);
  if (e != cudaSuccess) return e;
  if (!given && (e = run_stats(s, x, xr, wimg, lse, px, status, st)) != cudaSuccess) return e;
  return run_slice(s, s0.G, x, f, xr, fr, wimg, px, tokens, wsum, finalize, part, status, st);
}

cudaError_t tc_slice_fwd(const Shape& s0, const void* x, const void* f, const float* W, const float* bias,
                         const float* tau, float* tokens, float* wsum, float* lse, int finalize, float* part,
                         void* prep, bool reset, uint32_t* status, cudaStream_t st) {
  return slice_with_prep(s0, x, f, W, bias, tau, tokens, wsum, lse, nullptr, finalize, part, prep, reset, status, st);
}

cudaError_t tc_slice_fwd_lse(const Shape& s0, const void* x, const void* f, const float* W, const float* bias,
                             const float* tau, const float* lse, float* tokens, float* wsum, int finalize,
                             float* part, void* prep, bool reset, uint32_t* status, cudaStream_t st) {
  return slice_with_prep(s0, x, f, W, bias, tau, tokens, wsum, nullptr, lse, finalize, part, prep, reset, status, st);
}

// The slice on prepared operands: the W image and the point-extra rows at px; xr and
// fr the residual halves of x and fx (X3), else null.
cudaError_t run_slice(const Shape& s, int G, const void* x, const void* f, const void* xr, const void* fr,
                      const uint8_t* wimg, void* px, float* tokens, float* wsum, int finalize, float* part,
                      uint32_t* status, cudaStream_t st) {
  cudaError_t e;
  const bool x3 = xr != nullptr;
  CUtensorMap xmap, fmap, pmap, xrmap, frmap;
  if (!make_point_map(&xmap, x, s, kD, CU_TENSOR_MAP_SWIZZLE_64B)) return cudaErrorInvalidValue;
  if (!make_point_map(&fmap, f, s, 16, CU_TENSOR_MAP_SWIZZLE_32B)) return cudaErrorInvalidValue;
  if (!make_px_map(&pmap, px, s.BH(), padded_n(s))) return cudaErrorInvalidValue;
  if (!make_point_map(&xrmap, x3 ? xr : x, s, kD, CU_TENSOR_MAP_SWIZZLE_64B)) return cudaErrorInvalidValue;
  if (!make_point_map(&frmap, x3 ? fr : f, s, 16, CU_TENSOR_MAP_SWIZZLE_32B)) return cudaErrorInvalidValue;
  const int R = slice_blocks(s), P = slice_splits(s);
  dim3 grid((unsigned)R, (unsigned)P, (unsigned)s.BH());
  const size_t sm = smem_slice(x3);
  const auto kernel = x3 ? k_slice<true, true> : (s.dot == FS_DOT_BF16X2 ? k_slice<true, false> : k_slice<false, false>);
  if ((e = set_smem(kernel, sm)) != cudaSuccess) return e;
  if ((e = launch(kernel, grid, dim3(kThreads), sm, st, xmap, fmap, pmap, xrmap, frmap, wimg, part, s.N, padded_n(s),
                  s.H, s.G, P, status)) != cudaSuccess) return e;
  Shape so = s;
  so.G = G;
  return simt_reduce_tokens(so, P, part, s.G, tokens, wsum, finalize, st);
}

cudaError_t tc_deslice_fwd(const Shape& s0, const void* x, const float* W, const float* bias, const float* tau,
                           const float* zp, const float* lse, void* out, void* prep, bool reset, uint32_t* status,
                           cudaStream_t st) {
  const Shape s = tc_padded(s0);
  const bool x3 = x3_shape(s);
  const X3Ranges xr = x3_ranges(s0);
  uint8_t* wimg = static_cast<uint8_t*>(prep);
  uint8_t* zimg = wimg + align_up(w_image_bytes(s), 256);
  uint8_t* px = zimg + align_up(z_image_bytes(s), 256);
  uint8_t* xh = px + align_up(px_bytes(s), 256);
  // With split products the z' image holds z' hi then its residual (G*128 bytes per (b,h)).
  Prepare p(s, s0.G, tau, status, reset);
  p.weights(W, bias, wimg);
  p.tokens(zp, nullptr, zimg, x3);
  p.rows(lse, px);
  if (x3) p.split(s, x, xh, half_bytes(s));
  cudaError_t e = p.run(st);
  if (e != cudaSuccess) return e;
  CUtensorMap xmap, pmap, xrmap;
  if (!make_point_map(&xmap, x3 ? xh : x, s, kD, CU_TENSOR_MAP_SWIZZLE_64B)) return cudaErrorInvalidValue;
  if (!make_point_map(&xrmap, x3 ? xh + half_bytes(s) : x, s, kD, CU_TENSOR_MAP_SWIZZLE_64B))
    return cudaErrorInvalidValue;
  if (!make_px_map(&pmap, px, s.BH(), padded_n(s))) return cudaErrorInvalidValue;
  const int P = point_splits(s, (int)s.BH(), s.G / kGC);
  const bool split = s.dot == FS_DOT_BF16X2 || x3;
  const bool ps = x3;
  const bool hilo = split && smem_deslice(xr.size, true, 0, ps, x3) <= kMaxSmem;  // up to G = 768 (bf16)
  const size_t sm = smem_deslice(xr.size, hilo, 0, ps, x3);
  if (sm > kMaxSmem) return cudaErrorInvalidValue;
  const auto kernel = x3 ? k_deslice<0, true, true> : k_deslice<0, false>;
  if ((e = set_smem(kernel, sm)) != cudaSuccess) return e;
  for (int k = 0; k < xr.n; k++) {
    const int g0 = k * xr.size;
    if ((e = launch(kernel, dim3((unsigned)P, (unsigned)s.BH()), dim3(kDesl3Threads), sm, st, xmap,
                    pmap, xrmap, wimg, zimg, nullptr, static_cast<__nv_bfloat16*>(out), nullptr, nullptr, nullptr, nullptr, nullptr,
                    s.N, padded_n(s), s.H, s.G, g0, std::min(xr.size, s.G - g0), P, hilo ? 1 : 0,
                    (uint32_t)s.G * (ps ? 128 : 64), kStages, k > 0 ? 1 : 0, status)) != cudaSuccess) return e;
  }
  return cudaSuccess;
}

size_t tc_rows_smem(const Shape& s) { return smem_deslice(s.G, false, 2, true); }

cudaError_t tc_rows_bwd(const Shape& s, int Gi, int g0, int mode, const void* x, const uint8_t* wimg,
                        const uint8_t* zimg, const uint8_t* zimg2, const void* px, const void* v, const void* v2,
                        void* dfx, float* delta, float* wds, const float* dS, int accumulate, uint32_t* status,
                        cudaStream_t st) {
  const bool hilo = smem_deslice(s.G, true, mode, true) <= kMaxSmem;
  size_t sm = smem_deslice(s.G, hilo, mode, true);
  if (sm > kMaxSmem) return cudaErrorInvalidValue;
  int nst = kStages;
  if (mode == 3) {
    nst = std::min(kStages, 1 + (int)((kMaxSmem - sm) / kDStage));
    sm += (size_t)(nst - 1) * kDStage;
  }
  const int64_t Np = padded_n(s);
  CUtensorMap xmap, pmap;
  if (!make_point_map(&xmap, x, s, kD, CU_TENSOR_MAP_SWIZZLE_64B)) return cudaErrorInvalidValue;
  if (!make_px_map(&pmap, px, s.BH(), Np)) return cudaErrorInvalidValue;
  const int P = point_splits(s, (int)s.BH(), s.G / 64);
  dim3 grid((unsigned)P, (unsigned)s.BH());
  const auto kernel = mode == 1 ? k_deslice<1, true> : mode == 2 ? k_deslice<2, true> : k_deslice<3, true>;
  cudaError_t e = set_smem(kernel, sm);
  if (e != cudaSuccess) return e;
  return launch(kernel, grid, dim3(mode == 2 ? kThreads : kDesl3Threads), sm, st, xmap, pmap, xmap,
                wimg, zimg, zimg2, static_cast<__nv_bfloat16*>(dfx), static_cast<const __nv_bfloat16*>(v),
                static_cast<const __nv_bfloat16*>(v2), delta, wds, dS, s.N, Np, s.H, Gi, g0, s.G, P, hilo ? 1 : 0,
                (uint32_t)Gi * 128, nst, accumulate, status);
}

}  // namespace fs
