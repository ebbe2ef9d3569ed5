// Activations of the MXFP4 FFN kernel: a bf16 value as two e4m3 pieces that share a power-of-two scale per node and 32
// features, and where the pieces and scale bytes lie (see ffn.cu).  Used by the kernels that store the hidden states'
// pieces (routing.cu) and by the FFN kernel's epilogue.
#pragma once

#include <cuda_fp16.h>
#include <cuda_fp8.h>
#include <stdint.h>

namespace acm {

// Scales of a half-stage (64 features): two per row, up to 128 rows, in the order in which they go to tensor memory --
// rows i, i + 32, i + 64, i + 96 together, a word of each (the upper half of it unused).
constexpr int kMxActScaleBytes = 512;
__host__ __device__ inline int mx_scale_at(int row) { return (row & 31) * 16 + (row >> 5) * 4; }
constexpr int kMxPieceShift = 4;        // the second piece's scale is the first one's times 2^-4

// pieces of [H] features: H/64 half-stages of 2 n_pad <= 128 rows x 64 bytes, then their scales
__host__ __device__ inline size_t mx_act_scale_offset(int H) { return static_cast<size_t>(H / 64) * 128 * 64; }
__host__ __device__ inline size_t mx_act_bytes(int H) { return mx_act_scale_offset(H) + static_cast<size_t>(H / 64) * kMxActScaleBytes; }

// A block of 32 features of one node in pieces.  Within every eight features the order is 0 4 1 5 2 6 3 7: that of the
// unpacked weights (a packed word holds its eight codes in the order 0 2 4 6 1 3 5 7; its bytes' low nibbles come first).
struct MxBlock {
  uint32_t a[8], b[8];                 // e4m3, 32 of each
  unsigned char scale_a, scale_b;      // E8M0; 255 (NaN) if a value is not finite
};
__device__ __forceinline__ uint32_t mx_e4m3x2(float lo, float hi) {
  return __nv_cvt_float2_to_fp8x2(make_float2(lo, hi), __NV_SATFINITE, __NV_E4M3);
}
// w[i] = features 2 i (low half) and 2 i + 1 as bf16.  The scale puts the largest magnitude into [128, 256): a rounds to 4
// significand bits (at most 256, no saturation), the rest has at most 4 more and is at most 8, times 16.
__device__ __forceinline__ void mx_split_block(const uint32_t (&w)[16], MxBlock& out) {
  uint32_t m2 = 0u;                    // magnitudes order like their bits: the maximum of both halves at a time
#pragma unroll
  for (int i = 0; i < 16; ++i) m2 = __vmaxu2(m2, w[i] & 0x7fff7fffu);
  const uint32_t m = max(m2 & 0xffffu, m2 >> 16);
  const int scale = max(static_cast<int>(m >> 7) - 7, kMxPieceShift);
  const float mult = __int_as_float((254 - scale) << 23);
  constexpr float up = static_cast<float>(1 << kMxPieceShift);
#pragma unroll
  for (int g = 0; g < 8; ++g) {        // features 0 4 1 5 (g even) or 2 6 3 7 (g odd) of group g / 2
    uint32_t a2[2], b2[2];
    const uint32_t w0 = w[4 * (g / 2) + (g & 1)], w1 = w[4 * (g / 2) + (g & 1) + 2];
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const float y0 = __uint_as_float(j ? w0 & 0xffff0000u : w0 << 16) * mult;
      const float y1 = __uint_as_float(j ? w1 & 0xffff0000u : w1 << 16) * mult;
      a2[j] = mx_e4m3x2(y0, y1);
      const float2 back = __half22float2(__half2(__nv_cvt_fp8x2_to_halfraw2(static_cast<__nv_fp8x2_storage_t>(a2[j]), __NV_E4M3)));
      b2[j] = mx_e4m3x2((y0 - back.x) * up, (y1 - back.y) * up);
    }
    out.a[g] = a2[0] | (a2[1] << 16);
    out.b[g] = b2[0] | (b2[1] << 16);
  }
  const bool finite = m < 0x7f80u;
  out.scale_a = finite ? static_cast<unsigned char>(scale) : 255;
  out.scale_b = finite ? static_cast<unsigned char>(scale - kMxPieceShift) : 255;
}
// The pieces into rows ta and tb of a half-stage (rows of 64 bytes; block = 0 or 1 of the half-stage's two): 16-byte
// pieces at their place xor (row >> 1) & 3, the MMA's 64-byte swizzle.
__device__ __forceinline__ void mx_store_rows(unsigned char* rows, const MxBlock& k, int ta, int tb, int block) {
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const int c = 2 * block + i;
    *reinterpret_cast<uint4*>(rows + ta * 64 + ((c ^ ((ta >> 1) & 3)) << 4)) = make_uint4(k.a[4 * i], k.a[4 * i + 1], k.a[4 * i + 2], k.a[4 * i + 3]);
    *reinterpret_cast<uint4*>(rows + tb * 64 + ((c ^ ((tb >> 1) & 3)) << 4)) = make_uint4(k.b[4 * i], k.b[4 * i + 1], k.b[4 * i + 2], k.b[4 * i + 3]);
  }
}

}  // namespace acm
