// Activations of the MXFP4 FFN kernel: a bf16 value as three e5m2 pieces under a power-of-two scale per node and 32
// features (the second and third piece under its 2^-4 and 2^-8), and where the pieces and scale bytes lie (see ffn.cu).  Used by the kernels that store the hidden states'
// pieces (routing.cu) and by the FFN kernel's epilogue.
#pragma once

#include <cuda_fp16.h>
#include <cuda_fp8.h>
#include <stdint.h>
#include <string.h>

namespace acm {

constexpr int kMxPieces = 3;
constexpr int kMxPieceShift = 4;       // a piece's scale is that of the one before times 2^-4
// Scales of a half-stage (64 features): two bytes a node, up to 64 nodes, in the order in which they go to tensor memory --
// nodes i and i + 32 together, a word of each (the upper half of it unused).
constexpr int kMxActScaleBytes = 256;
__host__ __device__ inline int mx_scale_at(int node) { return (node & 31) * 8 + (node >> 5) * 4; }

// pieces of [H] features: H/64 half-stages of up to 3 x 64 rows x 64 bytes, then their scales
__host__ __device__ inline size_t mx_act_scale_offset(int H) { return static_cast<size_t>(H / 64) * (kMxPieces * 64 * 64); }
__host__ __device__ inline size_t mx_act_bytes(int H) { return mx_act_scale_offset(H) + static_cast<size_t>(H / 64) * kMxActScaleBytes; }

__host__ __device__ inline float mx_float(uint32_t bits) {
#ifdef __CUDA_ARCH__
  return __uint_as_float(bits);
#else
  float f;
  memcpy(&f, &bits, 4);
  return f;
#endif
}
// Scale of a block, w[i] = features 2 i (low half) and 2 i + 1 as bf16: its largest magnitude lies in [2^14, 2^15) of it.
// (E8M0, at least 8 = the third piece's shift; 255 = NaN if a value is not finite.)
__host__ __device__ inline int mx_block_scale(const uint32_t (&w)[16]) {
  uint32_t m = 0u;                     // magnitudes order like their bits
#ifdef __CUDA_ARCH__
#pragma unroll
  for (int i = 0; i < 16; ++i) m = __vmaxu2(m, w[i] & 0x7fff7fffu);
  m = max(m & 0xffffu, m >> 16);
#else
  for (int i = 0; i < 32; ++i) {
    const uint32_t v = (w[i / 2] >> (16 * (i & 1))) & 0x7fffu;
    m = v > m ? v : m;
  }
#endif
  const int above = static_cast<int>(m >> 7) - 14;
  constexpr int least = kMxPieceShift * (kMxPieces - 1);
  return m >= 0x7f80u ? 255 : above > least ? above : least;
}
// Features 16 i to 16 i + 15 of a block in pieces.  A bf16 has 8 significand bits, an e5m2 three: x = a + b + c, each the e5m2
// nearest to what the ones before leave (at most 2^-4 of the largest each time: below 2^15 under the next scale).  Exact for
// every |x| >= 2^-31 of the block's largest, off by at most 2^-39 of the largest below.  Within every eight features the order is 0 4 1 5 2 6 3 7: that of the unpacked weights (a packed word
// holds its eight codes in the order 0 2 4 6 1 3 5 7; its bytes' low nibbles come first).
__host__ __device__ __forceinline__ void mx_pieces(const uint32_t (&w)[16], int i, int scale, uint32_t (&piece)[kMxPieces][4]) {
  const float mult = mx_float(static_cast<uint32_t>(254 - (scale > 253 ? 253 : scale)) << 23);
#pragma unroll
  for (int g = 4 * i; g < 4 * i + 4; ++g) {        // features 0 4 1 5 (g even) or 2 6 3 7 (g odd) of group g / 2
    const uint32_t pair[2] = {w[4 * (g / 2) + (g & 1)], w[4 * (g / 2) + (g & 1) + 2]};
    uint32_t out[kMxPieces] = {0u, 0u, 0u};
#pragma unroll
    for (int j = 0; j < 2; ++j) {                  // the two words' low halves, then their high ones
      float y0 = mx_float(j ? pair[0] & 0xffff0000u : pair[0] << 16) * mult;
      float y1 = mx_float(j ? pair[1] & 0xffff0000u : pair[1] << 16) * mult;
#pragma unroll
      for (int p = 0; p < kMxPieces; ++p) {
        const __nv_fp8x2_storage_t q = __nv_cvt_float2_to_fp8x2(make_float2(y0, y1), __NV_SATFINITE, __NV_E5M2);
        out[p] |= static_cast<uint32_t>(q) << (16 * j);
        if (p + 1 < kMxPieces) {
          const float2 back = __half22float2(__half2(__nv_cvt_fp8x2_to_halfraw2(q, __NV_E5M2)));
          y0 = (y0 - back.x) * static_cast<float>(1 << kMxPieceShift);
          y1 = (y1 - back.y) * static_cast<float>(1 << kMxPieceShift);
        }
      }
    }
#pragma unroll
    for (int p = 0; p < kMxPieces; ++p) piece[p][g - 4 * i] = out[p];
  }
}
// A block (0 or 1 of its half-stage) of node t: its pieces into rows t, n_pad + t and 2 n_pad + t of the half-stage (rows of 64
// bytes), 16 bytes at a time at their place xor (row >> 1) & 3, the MMA's 64-byte swizzle (n_pad is a multiple of 16), and
// its scale.
__device__ __forceinline__ void mx_store_block(unsigned char* rows, unsigned char* scales, const uint32_t (&w)[16], int t,
                                               int n_pad, int block) {
  const int scale = mx_block_scale(w);
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    uint32_t k[kMxPieces][4];
    mx_pieces(w, i, scale, k);
    const int at = t * 64 + (((2 * block + i) ^ ((t >> 1) & 3)) << 4);
#pragma unroll
    for (int p = 0; p < kMxPieces; ++p)
      *reinterpret_cast<uint4*>(rows + p * n_pad * 64 + at) = make_uint4(k[p][0], k[p][1], k[p][2], k[p][3]);
  }
  scales[mx_scale_at(t) + block] = static_cast<unsigned char>(scale);
}

}  // namespace acm
