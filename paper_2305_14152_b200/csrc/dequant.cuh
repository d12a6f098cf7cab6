// Register-level dequantization of packed 3-/4-bit codes to bf16.
//
// The packed row is a little-endian bit string with column j at bits
// [b*j, b*j+b).  A "unit" is 32 consecutive columns: 4 words for b=4, 3 words
// for b=3.  Codes are turned into bf16 two at a time without any
// integer-to-float conversion: a code placed in the low mantissa bits of a
// bf16 whose exponent makes one code step equal 1.0 reads as (bias + q), and
// subtracting the bf16 constant (bias + z) gives (q - z) exactly (|q - z| <= 15).
//   code at mantissa bit 0 : bias 128 (bf16 0x4300)
//   code at mantissa bit 4 : bias 8   (bf16 0x4100)
// One 32-bit window of the bit string therefore yields the pair
// (column k, column k+4): b=4 has them 16 bits apart already, b=3 has them 12
// bits apart, so the window starts 4 bits early and the low code lands on
// mantissa bit 4.
#pragma once

#include <cuda_bf16.h>
#include <stdint.h>

namespace peqa {
namespace dq {

__device__ __forceinline__ uint32_t lop3_and_or(uint32_t x, uint32_t mask, uint32_t orv) {
  uint32_t r;
  asm("lop3.b32 %0, %1, %2, %3, 0xEA;" : "=r"(r) : "r"(x), "r"(mask), "r"(orv));  // (x & mask) | orv
  return r;
}

__device__ __forceinline__ uint32_t bf162_sub(uint32_t a, uint32_t b) {
  __nv_bfloat162 x = *reinterpret_cast<__nv_bfloat162*>(&a);
  __nv_bfloat162 y = *reinterpret_cast<__nv_bfloat162*>(&b);
  __nv_bfloat162 r = __hsub2(x, y);
  return *reinterpret_cast<uint32_t*>(&r);
}

__device__ __forceinline__ uint32_t bf162_mul(uint32_t a, uint32_t b) {
  __nv_bfloat162 x = *reinterpret_cast<__nv_bfloat162*>(&a);
  __nv_bfloat162 y = *reinterpret_cast<__nv_bfloat162*>(&b);
  __nv_bfloat162 r = __hmul2(x, y);
  return *reinterpret_cast<uint32_t*>(&r);
}

__device__ __forceinline__ uint32_t bf162_fma(uint32_t a, uint32_t b, uint32_t c) {
  __nv_bfloat162 x = *reinterpret_cast<__nv_bfloat162*>(&a);
  __nv_bfloat162 y = *reinterpret_cast<__nv_bfloat162*>(&b);
  __nv_bfloat162 z = *reinterpret_cast<__nv_bfloat162*>(&c);
  __nv_bfloat162 r = __hfma2(x, y, z);
  return *reinterpret_cast<uint32_t*>(&r);
}

__device__ __forceinline__ uint32_t bf162_broadcast(float s) {
  __nv_bfloat162 r = __float2bfloat162_rn(s);
  return *reinterpret_cast<uint32_t*>(&r);
}

// bf16x2 constant (bias_lo + z, bias_hi + z) matching pair_raw<BITS>().
template <int BITS>
__device__ __forceinline__ uint32_t zero_const(uint32_t z) {
  if (BITS == 4) return (0x4300u | z) * 0x00010001u;
  return ((0x4300u | z) << 16) | (0x4100u | (z << 4));
}

// 32-bit window of the 96-bit string (w0 lowest) starting at bit START
// (START may be negative: the string is shifted left).  Only bits 4..6 and
// 16..18 of the result are used by the caller.
template <int START>
__device__ __forceinline__ uint32_t window3(const uint32_t (&w)[3]) {
  if constexpr (START < 0) {
    return w[0] << (-START);
  } else {
    constexpr int a = START / 32;
    constexpr int sh = START % 32;
    if constexpr (sh == 0) {
      return w[a];
    } else if constexpr (sh + 19 <= 32 || a == 2) {
      return w[a] >> sh;
    } else {
      return __funnelshift_r(w[a], w[a + 1], sh);
    }
  }
}

// Biased bf16x2 of columns (K0, K0+4) of a unit, K0 = 8*blk + e, e in 0..3.
template <int BITS, int K0>
__device__ __forceinline__ uint32_t pair_raw(const uint32_t (&w)[BITS]) {
  if constexpr (BITS == 4) {
    constexpr int word = K0 / 8;
    constexpr int e = K0 % 8;
    return lop3_and_or(w[word] >> (4 * e), 0x000F000Fu, 0x43004300u);
  } else {
    return lop3_and_or(window3<3 * K0 - 4>(w), 0x00070070u, 0x43004100u);
  }
}

__device__ __forceinline__ uint32_t prmt(uint32_t a, uint32_t b, uint32_t sel) {
  uint32_t r;
  asm("prmt.b32 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "r"(sel));
  return r;
}

// Natural column order: the pair (2i, 2i + 1) of a block of 8 columns.  A block is whole bytes (4 or 3) of the string.  With the
// string and a copy shifted right by four bits every code lies within bits 0 to 6 of some byte of one of them, so one
// byte permutation puts both bytes of a pair in place and one logic operation leaves the biased pair: nine integer
// operations for eight codes.  (Pairs four columns apart, put in order by a permutation afterwards, took twelve; us, before / with this: forward of 40 tokens
// at 2048 x 2048 6.52 / 6.39, of 200 at 22016 x 8192 97.4 / 96, dX of 77 at 4096 x 4096 11.55 / 11.36.)
//   4 bits: column 2i in byte i of the word, 2i + 1 in byte i of the copy, both at bit 0 (bias 128)
//   3 bits: columns 0 1 | 2 3 | 4 5 | 6 7 at bits (0, 3) | (2 of the copy, 1) | (4, 3 of the copy) | (2, 1 of the copy);
//   a code at bit o has the bias 2^(7 - o)
__host__ __device__ constexpr int natural_kinds(int bits) { return bits == 4 ? 1 : 3; }           // pairs that differ in their biases
__host__ __device__ constexpr int natural_kind(int bits, int i) { return bits == 4 ? 0 : i == 0 ? 0 : i == 2 ? 2 : 1; }

template <int BITS>
__device__ __forceinline__ void natural_zero_consts(uint32_t z, uint32_t (&zc)[natural_kinds(BITS)]) {
  if constexpr (BITS == 4) {
    zc[0] = z * 0x00010001u + 0x43004300u;
  } else {
    zc[0] = z * 0x00080001u + 0x41804300u;
    zc[1] = z * 0x00020004u + 0x42804200u;
    zc[2] = z * 0x00080010u + 0x41804100u;
  }
}

// The four biased pairs of block BLK of a unit.
template <int BITS, int BLK>
__device__ __forceinline__ void block8_raw(const uint32_t (&w)[BITS], uint32_t (&x)[4]) {
  if constexpr (BITS == 4) {
    const uint32_t v = w[BLK], c = v >> 4;
    x[0] = lop3_and_or(prmt(v, c, 0x4400u), 0x000F000Fu, 0x43004300u);
    x[1] = lop3_and_or(prmt(v, c, 0x5511u), 0x000F000Fu, 0x43004300u);
    x[2] = lop3_and_or(prmt(v, c, 0x6622u), 0x000F000Fu, 0x43004300u);
    x[3] = lop3_and_or(prmt(v, c, 0x7733u), 0x000F000Fu, 0x43004300u);
  } else {
    constexpr int at = 24 * BLK + 4;                        // first bit of the copy
    uint32_t c;
    if constexpr (at % 32 + 20 <= 32) c = w[at / 32] >> (at % 32);
    else c = __funnelshift_r(w[at / 32], w[at / 32 + 1], at % 32);
    constexpr int b0 = 3 * BLK, b1 = b0 + 1, b2 = b0 + 2;   // the block's bytes
    // selectors: byte b % 4 of the word in the halves that take it (0 to 3), byte 4 + i of the copy in the others
    x[0] = lop3_and_or(prmt(w[b0 / 4], c, (b0 % 4) * 0x1111u), 0x00380007u, 0x41804300u);
    x[1] = lop3_and_or(prmt(w[b1 / 4], c, (b1 % 4) * 0x1100u + 0x0044u), 0x000E001Cu, 0x42804200u);
    x[2] = lop3_and_or(prmt(w[b1 / 4], c, (b1 % 4) * 0x0011u + 0x5500u), 0x00380070u, 0x41804100u);
    x[3] = lop3_and_or(prmt(w[b2 / 4], c, (b2 % 4) * 0x0011u + 0x6600u), 0x000E001Cu, 0x42804200u);
  }
}

// One block of 8 columns -> 4 bf16x2 registers in natural column order
// (out[0] = columns 0,1 ... out[3] = columns 6,7 of the block).
template <int BITS, int BLK, bool FOLD>
__device__ __forceinline__ void block8_natural(const uint32_t (&w)[BITS], const uint32_t (&zc)[natural_kinds(BITS)], uint32_t s2,
                                               uint32_t* out) {
  uint32_t x[4];
  block8_raw<BITS, BLK>(w, x);
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    out[i] = bf162_sub(x[i], zc[natural_kind(BITS, i)]);
    if (FOLD) out[i] = bf162_mul(out[i], s2);
  }
}

// A unit of 32 columns -> 16 bf16x2 registers holding (q - z) [* bf16(s) when
// FOLD] in natural column order.
template <int BITS, bool FOLD>
__device__ __forceinline__ void unit32_natural(const uint32_t (&w)[BITS], uint32_t z, float s,
                                               uint32_t (&out)[16]) {
  uint32_t zc[natural_kinds(BITS)];
  natural_zero_consts<BITS>(z, zc);
  const uint32_t s2 = FOLD ? bf162_broadcast(s) : 0u;
  block8_natural<BITS, 0, FOLD>(w, zc, s2, out + 0);
  block8_natural<BITS, 1, FOLD>(w, zc, s2, out + 4);
  block8_natural<BITS, 2, FOLD>(w, zc, s2, out + 8);
  block8_natural<BITS, 3, FOLD>(w, zc, s2, out + 12);
}

// Splits a real-valued zero-point into the integer the exact dequantization can use and
// the remainder the affine form carries: zi = clamp(rint(z), 0, 2^BITS - 1), delta = z - zi.
template <int BITS>
__device__ __forceinline__ void split_zero_point(float z, uint32_t& zi, float& delta) {
  const float r = fminf(fmaxf(rintf(z), 0.0f), (float)((1 << BITS) - 1));
  zi = (uint32_t)r;
  delta = z - r;
}

// A unit of 32 columns with a real-valued zero-point z = zi + delta (App. K trains z; its bits are handed in):
//   s*(q - z) = (q - zi)*s + c,  c = -delta*s,
// formed as one fused multiply-add per pair on the exact integers q - zi, so the operand is
// the product rounded once (with s and c rounded to bf16 first, as for grouped scales).
template <int BITS>
__device__ __forceinline__ void unit32_affine(const uint32_t (&w)[BITS], uint32_t z_bits, float s, uint32_t (&out)[16]) {
  uint32_t zi;
  float delta;
  split_zero_point<BITS>(__uint_as_float(z_bits), zi, delta);
  const float c = -delta * s;
  uint32_t zc[natural_kinds(BITS)];
  natural_zero_consts<BITS>(zi, zc);
  const uint32_t s2 = bf162_broadcast(s), c2 = bf162_broadcast(c);
  uint32_t x[4][4];
  block8_raw<BITS, 0>(w, x[0]);
  block8_raw<BITS, 1>(w, x[1]);
  block8_raw<BITS, 2>(w, x[2]);
  block8_raw<BITS, 3>(w, x[3]);
#pragma unroll
  for (int i = 0; i < 16; ++i)
    out[i] = bf162_fma(bf162_sub(x[i / 4][i % 4], zc[natural_kind(BITS, i % 4)]), s2, c2);
}

// ---------------------------------------------------------------------------
// Pairing for kernels whose contraction order is free (the streaming decode
// kernel: the activations are staged in whatever order the weights come out).
//
// A 3-bit code fits the 7 mantissa bits of a bf16 at any start bit p in 0..4,
// and with the exponent chosen so that one code step is 1.0 it reads as
// 2^(7-p) + q.  So one shifted window of the packed string can yield TWO pairs
// with two logic operations: with column A at bit 4 it holds
//   (A    at bit 4,  bias 8)   with  (A + 4 at bit 16, bias 128)   "std"
//   (A - 1 at bit 1, bias 64)  with  (A + 5 at bit 19, bias 16)    "alt"
// and a lone pair six columns apart can be taken as (bit 1, bit 19).  The 32
// columns of a unit split into six such double windows and four single ones
// (ten shifts, one of them by zero, and sixteen logic operations instead of
// sixteen of each).  Pair k of the unit, k = 0..15, is (stream_lo(k), stream_hi(k)); MMA
// m of the unit takes pairs 2m and 2m + 1.  4-bit codes have no second start
// position in a bf16 mantissa: their pairs stay (8b + e, 8b + e + 4).
// ---------------------------------------------------------------------------
// windows: A = 1, A = 3, (4,10), (9,13), A = 12, A = 15, (18,22), (21,27), A = 24, A = 26
__host__ __device__ constexpr int stream_lo(int bits, int k) {
  constexpr int lo3[16] = {1, 0, 3, 2, 4, 9, 12, 11, 15, 14, 18, 21, 24, 23, 26, 25};
  return bits == 3 ? lo3[k] : 8 * (k / 4) + k % 4;
}
__host__ __device__ constexpr int stream_hi(int bits, int k) {
  constexpr int hi3[16] = {5, 6, 7, 8, 10, 13, 16, 17, 19, 20, 22, 27, 28, 29, 30, 31};
  return bits == 3 ? hi3[k] : 8 * (k / 4) + k % 4 + 4;
}
// "alt" pairs sit at bits (1, 19) of their window and carry the biases (64, 16); the others
// sit at bits (4, 16) and carry (8, 128).  4-bit pairs carry (128, 128).
__host__ __device__ constexpr bool stream_alt(int bits, int k) {
  constexpr bool alt3[16] = {false, true, false, true, true, false, false, true,
                             false, true, false, true, false, true, false, true};
  return bits == 3 ? alt3[k] : false;
}
__host__ __device__ constexpr uint32_t stream_alt_mask3() {
  uint32_t m = 0;
  for (int k = 0; k < 16; ++k) m |= (stream_alt(3, k) ? 1u : 0u) << k;
  return m;
}

// 32-bit window of the 96-bit string starting at bit START (may be -1), of which bits
// 0..21 are used.
template <int START>
__device__ __forceinline__ uint32_t window3_wide(const uint32_t (&w)[3]) {
  if constexpr (START < 0) {
    return w[0] << (-START);
  } else {
    constexpr int a = START / 32;
    constexpr int sh = START % 32;
    if constexpr (sh == 0) {
      return w[a];
    } else if constexpr (sh + 22 <= 32 || a == 2) {
      return w[a] >> sh;
    } else {
      return __funnelshift_r(w[a], w[a + 1], sh);
    }
  }
}

// The two biased bf16x2 registers of MMA M (pairs 2M and 2M + 1) of a unit.
template <int BITS, int M>
__device__ __forceinline__ void mma_pairs_stream(const uint32_t (&w)[BITS], uint32_t& p0,
                                                 uint32_t& p1) {
  if constexpr (BITS == 4) {
    // pairs (8b + e, +4) and (8b + e + 1, +4) with b = M / 2, e = 2 * (M % 2)
    p0 = pair_raw<4, 8 * (M / 2) + 2 * (M % 2)>(w);
    p1 = pair_raw<4, 8 * (M / 2) + 2 * (M % 2) + 1>(w);
  } else {
    constexpr uint32_t kStdMask = 0x00070070u, kStdMagic = 0x43004100u;   // bits 4-6 | 16-18
    constexpr uint32_t kAltMask = 0x0038000Eu, kAltMagic = 0x41804280u;   // bits 1-3 | 19-21
    constexpr int k0 = 2 * M, k1 = 2 * M + 1;
    if constexpr (!stream_alt(3, k0) && stream_alt(3, k1) &&
                  stream_lo(3, k1) == stream_lo(3, k0) - 1) {
      // a double window: column lo[k0] at bit 4
      const uint32_t x = window3_wide<3 * stream_lo(3, k0) - 4>(w);
      p0 = lop3_and_or(x, kStdMask, kStdMagic);
      p1 = lop3_and_or(x, kAltMask, kAltMagic);
    } else {
      // two single windows
      if constexpr (stream_alt(3, k0))
        p0 = lop3_and_or(window3_wide<3 * stream_lo(3, k0) - 1>(w), kAltMask, kAltMagic);
      else
        p0 = lop3_and_or(window3_wide<3 * stream_lo(3, k0) - 4>(w), kStdMask, kStdMagic);
      if constexpr (stream_alt(3, k1))
        p1 = lop3_and_or(window3_wide<3 * stream_lo(3, k1) - 1>(w), kAltMask, kAltMagic);
      else
        p1 = lop3_and_or(window3_wide<3 * stream_lo(3, k1) - 4>(w), kStdMask, kStdMagic);
    }
  }
}

// ---------------------------------------------------------------------------
// fp16 operands without a bias (the prepared decode).  A code in the ten mantissa bits of an fp16 whose
// exponent bits are zero is the subnormal q * 2^(o - 24), o being its lowest bit: the tensor core takes
// it exactly, so one logic operation per pair is all there is, no exponent to put in and no bias to take
// off the sums.  Three-bit codes fit at o = 0..7, four-bit codes at 0..6, in either half of a window, so
// a shift serves up to three pairs: 16 logic operations and 5 shifts for 32 three-bit codes, 16 and 4 for
// four-bit ones (the bf16 pairs above: 16 and 10, 16 and 12).  The factor 2^o is taken out of the
// activation the code meets, which is exact as long as that stays a normal number.
// A string's pairs 0..7 hold its columns 0..15 and pairs 8..15 its columns 16..31, so that two runs of
// 32 columns of the matrix make eight pairs of every lane.
// ---------------------------------------------------------------------------
__host__ __device__ constexpr int f16_lo_bit(int bits, int j) {
  constexpr int lo3[16] = {0, 3, 6, 9, 12, 15, 36, 39, 42, 45, 54, 66, 69, 72, 75, 78};
  return bits == 3 ? lo3[j] : 32 * (j / 4) + 4 * (j % 4);
}
__host__ __device__ constexpr int f16_hi_bit(int bits, int j) {
  constexpr int hi3[16] = {18, 21, 24, 27, 30, 33, 48, 51, 57, 60, 63, 81, 84, 87, 90, 93};
  return bits == 3 ? hi3[j] : f16_lo_bit(4, j) + 16;
}
// first bit of the pair's 32-bit window of the string
__host__ __device__ constexpr int f16_window(int bits, int j) {
  constexpr int win3[16] = {0, 0, 4, 4, 10, 10, 32, 32, 38, 38, 47, 64, 64, 71, 71, 71};
  return bits == 3 ? win3[j] : 32 * (j / 4) + 8 * (j % 4 / 2);
}
// places of the pair's codes in their fp16: the codes count 2^o
__host__ __device__ constexpr int f16_lo_o(int bits, int j) { return f16_lo_bit(bits, j) - f16_window(bits, j); }
__host__ __device__ constexpr int f16_hi_o(int bits, int j) { return f16_hi_bit(bits, j) - f16_window(bits, j) - 16; }
// a window that reaches into the next word needs a funnel shift; the same for all pairs of a window, so
// that they share it
__host__ __device__ constexpr bool f16_funnel(int bits, int j) {
  for (int k = 0; k < 16; ++k)
    if (f16_window(bits, k) == f16_window(bits, j) &&
        f16_hi_bit(bits, k) + bits > 32 * (f16_window(bits, j) / 32 + 1))
      return true;
  return false;
}
// string column (0..31) whose code lies at this bit of the string
__host__ __device__ constexpr int string_column(int bits, int bit) {
  for (int k = 0; k < 16; ++k) {
    if (bits * stream_lo(bits, k) == bit) return 2 * k;
    if (bits * stream_hi(bits, k) == bit) return 2 * k + 1;
  }
  return -1;
}
__host__ __device__ constexpr bool f16_pairs_ok(int bits) {
  uint32_t seen = 0u;
  for (int j = 0; j < 16; ++j) {
    const int lo = string_column(bits, f16_lo_bit(bits, j)), hi = string_column(bits, f16_hi_bit(bits, j));
    if (lo < 0 || hi < 0 || lo / 16 != j / 8 || hi / 16 != j / 8) return false;
    if (f16_lo_o(bits, j) < 0 || f16_lo_o(bits, j) + bits > 10) return false;
    if (f16_hi_o(bits, j) < 0 || f16_hi_o(bits, j) + bits > 10) return false;
    seen |= 1u << lo | 1u << hi;
  }
  return seen == 0xFFFFFFFFu;
}
static_assert(f16_pairs_ok(3) && f16_pairs_ok(4), "every column once, its code inside the mantissa");

// Pair J of a string as two fp16 subnormals.
template <int BITS, int J>
__device__ __forceinline__ uint32_t f16_pair(const uint32_t (&w)[BITS]) {
  constexpr int start = f16_window(BITS, J), a = start / 32, sh = start % 32;
  constexpr uint32_t m = (1u << BITS) - 1u;
  constexpr uint32_t mask = m << f16_lo_o(BITS, J) | m << (16 + f16_hi_o(BITS, J));
  uint32_t x;
  if constexpr (f16_funnel(BITS, J)) x = __funnelshift_r(w[a], w[a + 1], sh);
  else x = w[a] >> sh;
  return x & mask;
}

// ---------------------------------------------------------------------------
// Codes as unsigned bytes, for integer MMAs.  A code inside a byte of a word of the string, at bit o of it,
// is q * 2^o, so one AND makes four operands: 4-bit strings are eight ANDs for 32 codes, without a shift.
// Of a 3-bit string's 32 codes 24 lie inside a byte (six ANDs); the eight that straddle two are
// gathered into two words (two shifts and two logic operations each).  The factor 2^o is taken out of the
// activation the code meets, which keeps o bits less.  Register r (0..7) of a string, byte b, holds the code at position
// i8_pos, times 2^i8_o; registers 2j and 2j + 1 are one MMA's.  HALF: registers 0..3 hold the
// string's columns 0..15 and 4..7 its columns 16..31 (four byte permutations more for 3-bit strings).
// ---------------------------------------------------------------------------
__host__ __device__ constexpr int i8_pos(int bits, bool half, int r, int b) {
  if (bits == 4) return 8 * (r / 2) + 2 * b + (r & 1);
  constexpr int plain[8][4] = {{0, 3, 6, 8},     {1, 4, 7, 9},     {11, 14, 16, 19}, {12, 15, 17, 20},
                               {22, 24, 27, 30}, {23, 25, 28, 31}, {2, 5, 13, 10},   {18, 21, 29, 26}};
  constexpr int halves[8][4] = {{0, 3, 6, 8},     {1, 4, 7, 9},     {11, 2, 16, 5},   {12, 13, 17, 10},
                                {22, 24, 27, 30}, {23, 25, 28, 31}, {14, 18, 19, 21}, {15, 29, 20, 26}};
  return half ? halves[r][b] : plain[r][b];
}
__host__ __device__ constexpr int i8_o(int bits, bool half, int r, int b) {
  const int p = i8_pos(bits, half, r, b);
  if (bits == 4) return 4 * (p & 1);
  switch (p) {                                     // the gathered ones
    case 2: case 10: case 13: case 18: case 26: case 29: return 0;
    case 5: case 21: return 1;
    default: return 3 * p % 8;
  }
}
// string column of the code at position p
__host__ __device__ constexpr int position_column(int bits, bool canon, int p) {
  return canon ? p : string_column(bits, bits * p);
}
__host__ __device__ constexpr bool i8_ok(int bits, bool half) {
  uint32_t seen = 0u;
  for (int r = 0; r < 8; ++r)
    for (int b = 0; b < 4; ++b) {
      const int p = i8_pos(bits, half, r, b);
      if (i8_o(bits, half, r, b) + bits > 8) return false;
      if (half && string_column(bits, bits * p) / 16 != r / 4) return false;
      seen |= 1u << p;
    }
  return seen == 0xFFFFFFFFu;
}
static_assert(i8_ok(3, false) && i8_ok(3, true) && i8_ok(4, false) && i8_ok(4, true), "every code once, inside its byte");

template <int BITS, bool HALF>
__device__ __forceinline__ void i8_string(const uint32_t (&w)[BITS], uint32_t (&r)[8]) {
  if constexpr (BITS == 4) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      r[2 * j] = w[j] & 0x0F0F0F0Fu;
      r[2 * j + 1] = w[j] & 0xF0F0F0F0u;
    }
  } else {
    r[0] = w[0] & 0x071C0E07u;
    r[1] = w[0] & 0x38E07038u;
    const uint32_t l1 = w[1] & 0x0E071C0Eu, h1 = w[1] & 0x7038E070u;
    // positions 2, 5, 10 (bits 6, 15, 30) and 13 (bit 39); 18, 21, 26 (54, 63, 78) and 29 (87)
    const uint32_t s1 = lop3_and_or(w[1] << 9, 0x00070000u, __funnelshift_r(w[0], w[1], 6) & 0x07000E07u);
    const uint32_t s2 = lop3_and_or(w[2] >> 7, 0x00070000u, __funnelshift_r(w[1], w[2], 22) & 0x07000E07u);
    if constexpr (HALF) {
      r[2] = prmt(l1, s1, 0x5240u);
      r[3] = prmt(h1, s1, 0x7260u);
      r[4] = w[2] & 0x1C0E071Cu;
      r[5] = w[2] & 0xE07038E0u;
      r[6] = prmt(l1, s2, 0x5341u);
      r[7] = prmt(h1, s2, 0x7361u);
    } else {
      r[2] = l1;
      r[3] = h1;
      r[4] = w[2] & 0x1C0E071Cu;
      r[5] = w[2] & 0xE07038E0u;
      r[6] = s1;
      r[7] = s2;
    }
  }
}

}  // namespace dq
}  // namespace peqa
