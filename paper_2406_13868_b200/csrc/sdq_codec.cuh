// Device-side number-format helpers of the packer and the activation quantizer.
// E2M1 / E4M3 encoding uses the hardware converters (round to nearest even, saturate to the largest
// finite value); scales are powers of two so every scaling below is exact.
#pragma once
#include <cuda_bf16.h>
#include <cuda_fp4.h>
#include <cuda_fp8.h>
#include <stdint.h>

namespace sdq {

__device__ __forceinline__ float bf16_bits_to_float(uint32_t h) { return __uint_as_float(h << 16); }

// a = f * 2^p with f in [1, 2):  returns p and f (a > 0, finite; subnormals handled)
__device__ __forceinline__ void split_pow2(float a, int& p, float& f) {
  p = ilogbf(a);
  f = scalbnf(a, -p);
}

// E8M0 code of the Q-Vector scale of 4-bit values whose largest magnitude is amax
//   rule 0: E = floor(log2 amax) - 2      rule 1: E = smallest integer with amax <= 6 * 2^E
__device__ __forceinline__ uint32_t e8m0_scale_code(float amax, int rule) {
  if (amax == 0.0f) return 0u;
  int p;
  float f;
  split_pow2(amax, p, f);
  int E = (rule == 0) ? (p - 2) : ((f <= 1.5f) ? (p - 2) : (p - 1));
  int c = E + 127;
  return (uint32_t)min(max(c, 0), 254);
}

// the same from the bit pattern of a non-negative finite bf16: with exponent field E the floor rule gives E - 2, and the
// smallest E with amax <= 6 * 2^E is one more when the significand exceeds 1.5; zeros and subnormals end at code 0 either way
__device__ __forceinline__ uint32_t e8m0_scale_code_bf16(uint32_t key, bool ceil_rule) {
  const int c = (int)(key >> 7) - 2 + ((ceil_rule && (key & 127u) > 64u) ? 1 : 0);
  return (uint32_t)max(c, 0);
}

// int8 operands (Section 5.1: W_o and A_o in int8): scale amax / 127 (1 for an all-zero vector) and code = the integer
// nearest to x / s, ties to even, limited to +-127 -- both quotients in fp32, IEEE round-to-nearest divisions, the
// precision in which the code is decided; returns the code's byte
__device__ __forceinline__ float int8_scale(float amax) { return amax == 0.0f ? 1.0f : __fdiv_rn(amax, 127.0f); }
__device__ __forceinline__ uint32_t int8_code(float x, float s) {
  const float r = fminf(fmaxf(rintf(__fdiv_rn(x, s)), -127.0f), 127.0f);
  return (uint32_t)(int)r & 0xFFu;
}

// The same code for a whole vector without a division per element: inv = 1 / s.  x * inv is within 2.3e-5 of the fp32
// quotient RN(x / s) (two roundings of 2^-24 against one, at most 127), so unless it lies within 2^-14 of a half-integer both
// round to the same integer; otherwise (one element in 8000), or where 1 / s leaves the normal range, the quotient
// itself decides.  Adding 1.5 * 2^23 rounds to the nearest even integer and leaves its two's complement in the low bits.
struct Int8Coder { float s, inv; bool exact; };
__device__ __forceinline__ Int8Coder int8_coder(float s) {
  Int8Coder c;
  c.s = s; c.inv = __fdiv_rn(1.0f, s); c.exact = !(s > 1e-30f);
  return c;
}
__device__ __forceinline__ uint32_t int8_code(float x, const Int8Coder& k) {
  const float q = x * k.inv, t = q + 12582912.0f;
  uint32_t c = __float_as_uint(t) & 0xFFu;
  if (k.exact || fabsf(q - (t - 12582912.0f)) > 0.5f - 6.103515625e-5f) c = int8_code(x, k.s);
  return c;
}

// exponent e of the power-of-two scale of an 8-bit (E4M3, max 448 = 1.75 * 2^8) operand:
// the smallest integer with amax <= 448 * 2^e, limited to what an E8M0 byte can carry
__device__ __forceinline__ int fp8_scale_exp(float amax) {
  if (amax == 0.0f) return 0;
  int p;
  float f;
  split_pow2(amax, p, f);
  int e = (f <= 1.75f) ? (p - 8) : (p - 7);
  return min(max(e, -127), 127);
}

// 2^(127 - c) for an E8M0 code c <= 253 and 2^(-e) for an 8-bit scale exponent e in [-127, 120], built from
// the exponent field: multiplying by them is exact (the products here never overflow; results too small for
// fp32 are far below half of the smallest E2M1 / E4M3 step and round to zero either way)
__device__ __forceinline__ float pow2_inv_e8m0(uint32_t c) { return __uint_as_float((254u - c) << 23); }
__device__ __forceinline__ float pow2_neg(int e) { return __uint_as_float((uint32_t)(127 - e) << 23); }

// Quotients x / y that are about to be rounded to a small format, without dividing: inv is 1 / y to within 2^-22 of it.  If
// x and (every rounding boundary) * y are integers below 256 times powers of two, the quotient either equals a boundary or is at
// least 1 / 255 of it away; x * inv is within 2^-21 of the quotient, so rounding it to 16 significant bits restores the
// boundaries and moves nothing across one.
__device__ __forceinline__ float small_quotient(float x, float inv) {
  return __uint_as_float((__float_as_uint(x * inv) + 0x80u) & 0xFFFFFF00u);
}
// Two-level scaling (SDQ_SCALE_UE4M3), on magnitudes already multiplied by 2^-t (pow2_neg): unsigned E4M3 code of the Q-Vector
// scale nearest to a / 6 (ties to even; 6 times an E4M3 midpoint has 8 significant bits), at least the smallest positive code
// unless a == 0
__device__ __forceinline__ uint32_t ue4m3_scale_code(float a, bool nonzero) {
  const uint32_t c = (uint32_t)__nv_cvt_float_to_fp8(small_quotient(a, 1.0f / 6.0f), __NV_SATFINITE, __NV_E4M3);
  return nonzero ? max(c, 1u) : 0u;
}
// 1 / scale of code c > 0 for small_quotient (an E4M3 value times an E2M1 boundary, 1, 3, 5 or 7 times a power of two, has 7
// significant bits)
__device__ __forceinline__ float ue4m3_scale_inverse(uint32_t c) {
  const __half_raw h = __nv_cvt_fp8_to_halfraw((__nv_fp8_storage_t)c, __NV_E4M3);
  return __fdividef(1.0f, __half2float(__half(h)));
}

// two packed bf16 times a power of two (the bits of a bf16), as floats, in one instruction each (unpacking and multiplying take
// two a pair more: 2048 x 11008 18.5 -> 18.0 us).  Rounded once, as the fp32 product is; the sum's -0 keeps the sign of zeros
__device__ __forceinline__ void scaled2(uint32_t x, uint32_t s, float& lo, float& hi) {
  asm("{\n.reg .b16 l, h, t;\n"
      "mov.b32 {l, h}, %2;\n"
      "cvt.u16.u32 t, %3;\n"
      "fma.rn.f32.bf16 %0, l, t, %4;\n"
      "fma.rn.f32.bf16 %1, h, t, %4;\n}"
      : "=f"(lo), "=f"(hi) : "r"(x), "r"(s), "f"(-0.0f));
}
// two floats -> two E2M1 codes in one byte (x in the low nibble)
__device__ __forceinline__ uint32_t e2m1x2(float x, float y) {
  return (uint32_t)__nv_cvt_float2_to_fp4x2(make_float2(x, y), __NV_E2M1, cudaRoundNearest);
}
// eight floats -> eight E2M1 codes in one word (the first in the lowest nibble)
__device__ __forceinline__ uint32_t e2m1x8(const float (&v)[8]) {
  uint32_t d;
  asm("{\n.reg .b8 a, b, c, d;\n"
      "cvt.rn.satfinite.e2m1x2.f32 a, %2, %1;\n"
      "cvt.rn.satfinite.e2m1x2.f32 b, %4, %3;\n"
      "cvt.rn.satfinite.e2m1x2.f32 c, %6, %5;\n"
      "cvt.rn.satfinite.e2m1x2.f32 d, %8, %7;\n"
      "mov.b32 %0, {a, b, c, d};\n}"
      : "=r"(d) : "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7]));
  return d;
}
// four floats -> four E4M3 codes in one word (the first in the lowest byte)
__device__ __forceinline__ uint32_t e4m3x4(float a, float b, float c, float d) {
  uint32_t w;
  asm("{\n.reg .b16 l, h;\n"
      "cvt.rn.satfinite.e4m3x2.f32 l, %2, %1;\n"
      "cvt.rn.satfinite.e4m3x2.f32 h, %4, %3;\n"
      "mov.b32 %0, {l, h};\n}"
      : "=r"(w) : "f"(a), "f"(b), "f"(c), "f"(d));
  return w;
}
// bytes of {b, a} picked by the four nibbles of sel (bit 3 of a nibble: the byte's sign bit, spread over it)
__device__ __forceinline__ uint32_t prmt(uint32_t a, uint32_t b, uint32_t sel) {
  uint32_t d;
  asm("prmt.b32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(sel));
  return d;
}
// two packed bf16, infinities as the largest finite number of their sign
__device__ __forceinline__ uint32_t finite2(uint32_t x) {
  const uint32_t top = 0x7F7F7F7Fu, bottom = 0xFF7FFF7Fu;
  const __nv_bfloat162 r = __hmin2(__hmax2(*reinterpret_cast<const __nv_bfloat162*>(&x), *reinterpret_cast<const __nv_bfloat162*>(&bottom)),
                                   *reinterpret_cast<const __nv_bfloat162*>(&top));
  return *reinterpret_cast<const uint32_t*>(&r);
}
// running maxima of two packed bf16 magnitudes; a NaN stays, as one above infinity
__device__ __forceinline__ uint32_t max_abs2(uint32_t m, uint32_t x) {
  const __nv_bfloat162 r = __hmax2_nan(*reinterpret_cast<const __nv_bfloat162*>(&m), __habs2(*reinterpret_cast<const __nv_bfloat162*>(&x)));
  return *reinterpret_cast<const uint32_t*>(&r);
}
// two floats -> two E4M3 codes in 16 bits (x in the low byte)
__device__ __forceinline__ uint32_t e4m3x2(float x, float y) {
  return (uint32_t)__nv_cvt_float2_to_fp8x2(make_float2(x, y), __NV_SATFINITE, __NV_E4M3);
}
__device__ __forceinline__ uint32_t e4m3x1(float x) { return (uint32_t)__nv_cvt_float_to_fp8(x, __NV_SATFINITE, __NV_E4M3); }

// selection keys of one S-Vector: the 15-bit magnitude itself, or -- with a per-input-channel weight c[k] -- the bit
// pattern of the fp32 product |w| * c[k] (one round-to-nearest multiply; non-negative floats order like their bits).
// Returns nonzero if a channel weight is negative, infinite or NaN.
__device__ __forceinline__ uint32_t selection_keys(const uint32_t (&key)[8], const float* __restrict__ colw, int g, uint32_t (&skey)[8]) {
  if (!colw) {
#pragma unroll
    for (int i = 0; i < 8; ++i) skey[i] = key[i];
    return 0;
  }
  const float4 c0 = reinterpret_cast<const float4*>(colw + 8 * g)[0], c1 = reinterpret_cast<const float4*>(colw + 8 * g)[1];
  const float c[8] = {c0.x, c0.y, c0.z, c0.w, c1.x, c1.y, c1.z, c1.w};
  uint32_t bad = 0;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    bad |= !(c[i] >= 0.0f && c[i] <= 3.4028234663852886e38f);
    skey[i] = __float_as_uint(__fmul_rn(bf16_bits_to_float(key[i]), c[i]));
  }
  return bad;
}
// significance of position i as a float (for the pair score)
__device__ __forceinline__ float key_value(uint32_t key, uint32_t skey, bool weighted) {
  return weighted ? __uint_as_float(skey) : bf16_bits_to_float(key);
}

// |x| with +-Inf replaced by the largest finite bf16 (saturation)
__device__ __forceinline__ float sat_abs(float x) { return fminf(fabsf(x), 3.3895313892515355e38f); }
__device__ __forceinline__ float sat(float x) { return copysignf(sat_abs(x), x); }

// ---- Stage 2 helpers shared by the tiled and the plain packer (one thread per S-Vector of 8 weights) ----------
// the 8 bf16 bit patterns of an S-Vector (one 16-byte load)
__device__ __forceinline__ void load_group(const __nv_bfloat16* w, uint32_t (&bits)[8]) {
  const uint4 v = *reinterpret_cast<const uint4*>(w);
  const uint32_t r[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    bits[2 * i] = r[i] & 0xFFFFu;
    bits[2 * i + 1] = r[i] >> 16;
  }
}

// positions of the out_n most (small: least) significant values, ties to the lower index
__device__ __forceinline__ void select_outliers(const uint32_t (&key)[8], int out_n, bool small, int& o0, int& o1) {
  o0 = o1 = -1;
  if (out_n >= 1) {
    int b = 0;
#pragma unroll
    for (int i = 1; i < 8; ++i)
      if (small ? key[i] < key[b] : key[i] > key[b]) b = i;
    o0 = b;
  }
  if (out_n >= 2) {
    int b = -1;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      if (i == o0) continue;
      if (b < 0 || (small ? key[i] < key[b] : key[i] > key[b])) b = i;
    }
    o1 = b;
    if (o0 > o1) { int t = o0; o0 = o1; o1 = t; }
  }
}

}  // namespace sdq
