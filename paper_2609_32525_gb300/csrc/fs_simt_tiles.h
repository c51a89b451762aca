// The tiled fp32 passes (fs_simt_tiles.cuh), one explicit instantiation per point type:
// fs_simt_f32.cu and fs_simt_bf16.cu.
#pragma once

#include "fs_internal.h"

namespace fs {

constexpr int kSimtTP = 128;  // points per tile of every tiled pass

// Slots per tile: small slice counts take the narrower tile (d = 64 has only the wide one).
inline int simt_tile_slots(const Shape& s) { return s.G <= 32 && s.d != 64 ? 32 : 64; }

// reset: this is the first launch of a call that knows the temperatures; it writes the status
// word (clear, or a bad temperature).
template <typename T>
struct SimtTiles {
  static cudaError_t stats(const Shape& s, const T* x, const float* W, const float* bias, const float* tau,
                           float* lse, bool reset, uint32_t* status, cudaStream_t st);
  static cudaError_t slice(const Shape& s, int P, const T* x, const T* f, const float* W, const float* bias,
                           const float* tau, const float* lse, float* part, bool reset, uint32_t* status,
                           cudaStream_t st);
  static cudaError_t deslice(const Shape& s, const T* x, const float* W, const float* bias, const float* tau,
                             const float* zp, const float* lse, T* out, bool reset, uint32_t* status,
                             cudaStream_t st);
  // mode 0: the deslice's backward (dO, z'); 1: the slice's (fx, dU | dS); 2: both at once.
  static cudaError_t backward(const Shape& s, int mode, int P, const T* x, const T* dO, const T* fx, const float* W,
                              const float* bias, const float* tau, const float* zp, const float* dUS,
                              const float* lse, T* dx, T* dfx, float* delta, float* dt_part, float* part,
                              int accumulate, bool reset, uint32_t* status, cudaStream_t st);
};

}  // namespace fs
