// The 4-bit code of 32 values of one channel block, as four plane words (Sec. 3.2, Eq. 2): c = clip(floor(k / s), -8, 7) + 8 with
// the stored scale s, bit i of word p = bit (3 - p) of value i's code.  Used by the plane builder and by the rotation that
// quantises its own accumulator.
//
// Two values at a time: n = round(k * (1/s)) by the 1.5 * 2^23 trick, d = k - n s in one fused multiply-add.  n s is exact in
// it (n has 4 bits, s 11), so the SIGN of d is exact and floor(k / s) = n - (d < 0) whatever the rounding of 1/s and of the
// product did: |k| <= 8.01 s (12 s where an eighth of the maximum was rounded to a subnormal s: clipped like the rest), so they
// move k / s by less than 1e-5 and n is one of the two integers next to it.  -0 counts as 0 (the negated n is +0 there, so d is +0).  The packed 16-bit add-min-relu clips both codes to 0..15 in one instruction,
// the codes are collected as nibbles, and two rounds of masked merges turn four registers of eight nibbles into the four
// plane words: about 4.5 instructions per value, against 13 for four compare-and-select steps with a predicated OR each.
#pragma once
#include "fathom_common.cuh"

__device__ __forceinline__ float2 fathom_fma2(float2 a, float2 b, float2 c) {
  float2 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;"
      : "=l"(reinterpret_cast<unsigned long long&>(d))
      : "l"(reinterpret_cast<const unsigned long long&>(a)), "l"(reinterpret_cast<const unsigned long long&>(b)),
        "l"(reinterpret_cast<const unsigned long long&>(c)));
  return d;
}

// sc: the stored scale, > 0 (a zero scale has no 1/s: the caller writes code 8 for every value); inv: 1 / sc
__device__ __forceinline__ void fathom_quantise32(const float (&v)[32], float sc, float inv, uint32_t (&w)[FATHOM_NPLANES]) {
  const float2 s2 = make_float2(sc, sc), inv2 = make_float2(inv, inv), minus1 = make_float2(-1.0f, -1.0f);
  const float2 magic = make_float2(12582912.0f + 8.0f, 12582912.0f + 8.0f);   // 1.5 * 2^23 + 8: the low bits of the sum are n + 8
  uint32_t nib[4] = {0u, 0u, 0u, 0u};                          // register r: nibble x = code of value 4 x + r
#pragma unroll
  for (int x = 3; x >= 0; --x) {                              // nibbles x and x + 4: the two 16-bit lanes
    float2 t[4], d[4];                                         // values 4 x .. 4 x + 3 and the four 16 further on
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int i = 4 * x + 2 * (e & 1) + 16 * (e >> 1);
      const float2 k = make_float2(v[i], v[i + 1]);
      t[e] = fathom_fma2(k, inv2, magic);
      d[e] = fathom_fma2(fathom_fma2(t[e], minus1, magic), s2, k);
    }
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const float t0 = r & 1 ? t[r >> 1].y : t[r >> 1].x, t1 = r & 1 ? t[2 + (r >> 1)].y : t[2 + (r >> 1)].x;
      const float d0 = r & 1 ? d[r >> 1].y : d[r >> 1].x, d1 = r & 1 ? d[2 + (r >> 1)].y : d[2 + (r >> 1)].x;
      const uint32_t n8 = __byte_perm(__float_as_uint(t0), __float_as_uint(t1), 0x5410);          // low halves: n + 8 each
      uint32_t below;                                          // 0xffff where d is negative
      asm("prmt.b32 %0, %1, %2, 0xffbb;" : "=r"(below) : "r"(__float_as_uint(d0)), "r"(__float_as_uint(d1)));
      nib[r] = (nib[r] << 4) | __viaddmin_s16x2_relu(n8, below, 0x000f000fu);
    }
  }
  // bit p of the codes: nibble x of word p = bits p of values 4 x .. 4 x + 3
  auto merge = [](uint32_t a, uint32_t b, uint32_t m) { return (a & m) | (b & ~m); };
  const uint32_t lo01 = merge(nib[0], nib[1] << 1, 0x55555555u), hi01 = merge(nib[0] >> 1, nib[1], 0x55555555u);
  const uint32_t lo23 = merge(nib[2], nib[3] << 1, 0x55555555u), hi23 = merge(nib[2] >> 1, nib[3], 0x55555555u);
  w[3] = merge(lo01, lo23 << 2, 0x33333333u);
  w[1] = merge(lo01 >> 2, lo23, 0x33333333u);
  w[2] = merge(hi01, hi23 << 2, 0x33333333u);
  w[0] = merge(hi01 >> 2, hi23, 0x33333333u);
}
