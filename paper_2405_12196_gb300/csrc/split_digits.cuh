// Digits of the error-free split (shared by the staged and the fused slice
// kernels). For an element x of a row with scale 2^e (|x| < 2^(e - 1)), the
// integer u = round(x 2^(8s - e)), |u| <= 2^(8s - 1), is written in balanced base
// 256, u = sum_{p < s} d_p 256^(s - 1 - p) with d_p in [-128, 127] (the leading
// one in [-128, 128]); slice p holds d_p 2^(-8p). The digits come from the FP64
// bit pattern with integer operations only.
#pragma once

#include <cuda_bf16.h>

#include "ytn_internal.hpp"

namespace ytn {

static_assert(kSlices == 6, "the digits are taken from fixed byte positions");

// The upper half of x as the float 2^23 + its value (one byte permute).
__device__ __forceinline__ float biased_short(uint32_t x) { return __uint_as_float(__byte_perm(x, 0x4B000000u, 0x7532u)); }

// Byte k of x as the float 2^23 + byte (one byte permute).
template <int K>
__device__ __forceinline__ float biased_byte(uint32_t x) {
  return __uint_as_float(__byte_perm(x, 0x4B000000u, 0x7540u | K));
}

// Two floats with at most 8 significant bits as a BF16 pair (low half: f0). Their
// BF16 values are exact: the upper 16 bits of each float.
__device__ __forceinline__ uint32_t pack_exact_bf16(float f0, float f1) {
  return __byte_perm(__float_as_uint(f0), __float_as_uint(f1), 0x7632u);
}

// Two FP32 multiply-adds in one instruction: (x0, x1) * m + a.
__device__ __forceinline__ void fma2(float &x0, float &x1, float m, float a) {
  asm("{\n\t.reg .b64 x, m, a;\n\tmov.b64 x, {%0, %1};\n\tmov.b64 m, {%2, %2};\n\tmov.b64 a, {%3, %3};\n\t"
      "fma.rn.f32x2 x, x, m, a;\n\tmov.b64 {%0, %1}, x;\n\t}"
      : "+f"(x0), "+f"(x1)
      : "f"(m), "f"(a));
}

// Eight consecutive elements of one row (raw FP64 bits; E: the row's largest biased
// exponent) -> s slices of 8 BF16 values each, packed as 16 bytes per slice (two
// elements per 32-bit word, the even one in the low half).
__device__ __forceinline__ void slice_digits8(const unsigned long long *bits8, int E, int s,
                                              uint32_t (&packed)[kSlices][4]) {
  // balanced base-256 digits: with T = |x| 2^(56 - e) < 2^55, whose integer digits start
  // at byte 6 (u = round(x 2^(8s - e)) has its last digit at byte 7 - s), and
  //   w = +-T + sum 128 256^b over the bytes b of the kept digits and the one below,
  // digit p is byte 6 - p of w minus 128, the leading one taking the carry above byte 6
  // as well (it lies in [-128, 128]). The 128 below the last digit rounds to nearest,
  // away from zero at a tie; for negative x the one's complement of T stands for -T:
  // ~T + 128 256^b + ... = (... - u) 256^(b+1) + a rest in [0, 256^(b+1)).
  const unsigned long long kHalves = 0x0080808080808080ull & (~0ull << (8 * (kSlices - s)));
#pragma unroll
  for (int j = 0; j < 8; j += 2) {
    uint32_t lo[2], hi[2];
#pragma unroll
    for (int h = 0; h < 2; h++) {
      const uint32_t xl = (uint32_t)bits8[j + h], xh = (uint32_t)(bits8[j + h] >> 32);
      const int Eb = (int)((xh >> 20) & 0x7FF);
      // |x| 2^(56 - e): the significand (53 bits), two bits up for a row's largest
      // elements and one place down for every exponent below theirs
      const uint32_t mh = (xh & 0xFFFFFu) | 0x100000u;
      uint32_t th = __funnelshift_l(xl, mh, 2), tl = xl << 2;
      int d = Eb != 0 ? E - Eb : 63;   // zero and subnormal elements give zero digits
      if (d >= 32) {
        tl = th;
        th = 0;
        d = min(d - 32, 31);   // th < 2^23: nothing left from 23 on
      }
      tl = __funnelshift_r(tl, th, d);
      th >>= d;
      const uint32_t sg = (uint32_t)((int)xh >> 31);
      const unsigned long long w = (((unsigned long long)(th ^ sg) << 32) | (tl ^ sg)) + kHalves;
      lo[h] = (uint32_t)w;
      hi[h] = (uint32_t)(w >> 32);
    }
    // slice p holds d_p 2^(-8p) = (byte - 128) 2^(-8p): from the float 2^23 + byte,
    // one exact FMA ((2^23 + byte) 2^(-8p) - (2^23 + 128) 2^(-8p), both terms and
    // the result representable); the leading digit (up to 256 - 128) from two bytes
    constexpr float kBias = 8388608.0f + 128.0f;
    auto put = [&](int p, float f0, float f1, float scale) {
      fma2(f0, f1, scale, -kBias * scale);
      packed[p][j >> 1] = pack_exact_bf16(f0, f1);
    };
    put(0, biased_short(hi[0]), biased_short(hi[1]), 1.0f);
    if (s > 1) put(1, biased_byte<1>(hi[0]), biased_byte<1>(hi[1]), 0x1p-8f);
    if (s > 2) put(2, biased_byte<0>(hi[0]), biased_byte<0>(hi[1]), 0x1p-16f);
    if (s > 3) put(3, biased_byte<3>(lo[0]), biased_byte<3>(lo[1]), 0x1p-24f);
    if (s > 4) put(4, biased_byte<2>(lo[0]), biased_byte<2>(lo[1]), 0x1p-32f);
    if (s > 5) put(5, biased_byte<1>(lo[0]), biased_byte<1>(lo[1]), 0x1p-40f);
  }
}

// Position of row rr's 16-byte chunk c (8 elements of K) inside a 128 x 32 slice:
// K-major, 64 bytes per row, chunk c stored at c ^ ((rr >> 1) & 3) (the 64-byte
// swizzle the tensor cores read).
__device__ __forceinline__ int slice_pos(int rr, int c) { return rr * 64 + ((c ^ ((rr >> 1) & 3)) << 4); }

__device__ __forceinline__ void store_slices(uint8_t *blk, int pos, int s, const uint32_t (&packed)[kSlices][4]) {
#pragma unroll
  for (int p = 0; p < kSlices; p++)
    if (p < s)   // slices beyond s are never read
      *reinterpret_cast<uint4 *>(blk + p * kSliceBytes + pos) =
          make_uint4(packed[p][0], packed[p][1], packed[p][2], packed[p][3]);
}

__device__ __forceinline__ int biased_exp(double x) { return (int)((__double_as_longlong(x) >> 52) & 0x7FF); }

}  // namespace ytn
