// gemm_epilogue.cuh -- the tensor-core GEMMs' fused epilogues (bias, residual,
// SwiGLU), shared by the few-row and the many-row kernel.
#pragma once

#include "kvr_internal.cuh"

namespace kvr {

// Epilogue for 16 consecutive rows t0..t0+15 of Y (the first `cnt` valid) at
// feature n of W.  All lanes of the warp call it together (SwiGLU exchanges
// lanes); every load is issued before any dependent use, so the chunk costs
// one L2 round trip, not sixteen.
template <class P>
__device__ __forceinline__ void epilogue16(const P &p, int t0, int n, const float *v, int cnt) {
  if (p.epi == GEMM_EPI_SWIGLU) {
    // rows 32b..32b+15 of W are gate, 32b+16..32b+31 up, of features
    // 16b..16b+15; lane = n % 32.  Lanes r and r ^ 16 swap their values, so
    // both hold gate and up of feature r % 16; the low half then writes the
    // even rows and the high half the odd ones.
    const int r = n & 31, hi = r >> 4;
    float o[16];
#pragma unroll
    for (int j = 0; j < 16; ++j) o[j] = __shfl_xor_sync(0xffffffffu, v[j], 16);
    __nv_bfloat16 *out = (__nv_bfloat16 *)p.out2 + (size_t)t0 * p.ld2 + (n >> 5) * 16 + (r & 15);
#pragma unroll
    for (int jj = 0; jj < 8; ++jj) {
      // low lanes hold gate in v, up in o; high lanes the reverse
      const float g = hi ? o[2 * jj + 1] : v[2 * jj], u = hi ? v[2 * jj + 1] : o[2 * jj];
      const int j = 2 * jj + hi;
      if (j < cnt) out[(size_t)j * p.ld2] = __float2bfloat16_rn(swiglu_bf16path(g, u));
    }
    return;
  }
  float *y = p.Y + (size_t)t0 * p.ldy + n;
  if (p.epi == GEMM_EPI_ACCUM) {
    float old[16];
#pragma unroll
    for (int j = 0; j < 16; ++j) old[j] = j < cnt ? y[(size_t)j * p.ldy] : 0.f;
#pragma unroll
    for (int j = 0; j < 16; ++j)
      if (j < cnt) y[(size_t)j * p.ldy] = old[j] + v[j];
    return;
  }
  float b = p.bias ? p.bias[n] : 0.f;
#pragma unroll
  for (int j = 0; j < 16; ++j)
    if (j < cnt) y[(size_t)j * p.ldy] = v[j] + b;
}

}  // namespace kvr
