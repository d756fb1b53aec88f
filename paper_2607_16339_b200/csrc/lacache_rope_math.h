// Rotation and storage-format arithmetic shared by the RoPE-on-write kernel, the
// projection's epilogue and the attention kernel's in-place rotation of a block's
// queries (Eq. 1): all must produce the same bits, so all call these.
#pragma once
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cstdint>

namespace lacache {

// 8 consecutive source features starting at element offset elem_off: fetched (N 16-byte words: fp32 takes two), and
// converted to fp32
template <int N>
__device__ __forceinline__ void rope_fetch8(const void* base, size_t elem_off, bool bf16_in, uint4 (&w)[N]) {
  if (bf16_in) {
    w[0] = *reinterpret_cast<const uint4*>(reinterpret_cast<const __nv_bfloat16*>(base) + elem_off);
  } else {
    const uint4* p = reinterpret_cast<const uint4*>(reinterpret_cast<const float*>(base) + elem_off);
#pragma unroll
    for (int i = 0; i < N; ++i) w[i] = p[i];
  }
}
template <int N>
__device__ __forceinline__ void rope_unpack8(const uint4 (&w)[N], bool bf16_in, float (&x)[8]) {
  if (bf16_in) {
    const __nv_bfloat162* p = reinterpret_cast<const __nv_bfloat162*>(&w[0]);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      float2 f = __bfloat1622float2(p[i]);
      x[2 * i] = f.x;
      x[2 * i + 1] = f.y;
    }
  } else {
    const float* p = reinterpret_cast<const float*>(&w[0]);
#pragma unroll
    for (int i = 0; i < 4 * N; ++i) x[i] = p[i];
  }
}
__device__ __forceinline__ void rope_load8(const void* base, size_t elem_off, bool bf16_in, float (&x)[8]) {
  uint4 w[2];
  rope_fetch8<2>(base, elem_off, bf16_in, w);
  rope_unpack8<2>(w, bf16_in, x);
}

// (x1, x2) = features (c, c + d/2) rotated by the angle whose cos / sin are given;
// separate roundings on purpose (no fma contraction)
__device__ __forceinline__ void rope_rotate8(const float (&x1)[8], const float (&x2)[8], const float (&cs)[8],
                                             const float (&sn)[8], float (&y1)[8], float (&y2)[8]) {
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    y1[i] = __fsub_rn(__fmul_rn(x1[i], cs[i]), __fmul_rn(x2[i], sn[i]));
    y2[i] = __fadd_rn(__fmul_rn(x2[i], cs[i]), __fmul_rn(x1[i], sn[i]));
  }
}

// 8 values as split bf16: hi = bf16(y), lo = bf16(y - hi), 16 bytes each
__device__ __forceinline__ void rope_split8(const float (&y)[8], uint4& hi, uint4& lo) {
  __nv_bfloat162* ph = reinterpret_cast<__nv_bfloat162*>(&hi);
  __nv_bfloat162* pl = reinterpret_cast<__nv_bfloat162*>(&lo);
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    __nv_bfloat16 h0 = __float2bfloat16_rn(y[2 * i]);
    __nv_bfloat16 h1 = __float2bfloat16_rn(y[2 * i + 1]);
    __nv_bfloat16 l0 = __float2bfloat16_rn(y[2 * i] - __bfloat162float(h0));
    __nv_bfloat16 l1 = __float2bfloat16_rn(y[2 * i + 1] - __bfloat162float(h1));
    ph[i] = __halves2bfloat162(h0, h1);
    pl[i] = __halves2bfloat162(l0, l1);
  }
}

// 8 values as fp16, saturated to the finite fp16 range (the storage format of V)
__device__ __forceinline__ uint4 rope_half8(const float (&y)[8]) {
  uint4 u;
  __half2* p = reinterpret_cast<__half2*>(&u);
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    float a = fminf(fmaxf(y[2 * i], -65504.f), 65504.f);
    float b = fminf(fmaxf(y[2 * i + 1], -65504.f), 65504.f);
    p[i] = __floats2half2_rn(a, b);
  }
  return u;
}

// 8 rotated values of q or k at element offset off of the tcgen05 engine's planes
__device__ __forceinline__ void rope_store8(void* hi_plane, void* lo_plane, size_t off, const float (&y)[8], bool f16) {
  if (f16) {   // one fp16 plane: the rotated value rounded once to fp16
    *reinterpret_cast<uint4*>(reinterpret_cast<__half*>(hi_plane) + off) = rope_half8(y);
    return;
  }
  uint4 uh, ul;
  rope_split8(y, uh, ul);
  *reinterpret_cast<uint4*>(reinterpret_cast<__nv_bfloat16*>(hi_plane) + off) = uh;
  // (plain operands keep the hi plane alone: the rotated value rounded once to bf16)
  if (lo_plane) *reinterpret_cast<uint4*>(reinterpret_cast<__nv_bfloat16*>(lo_plane) + off) = ul;
}

}  // namespace lacache
