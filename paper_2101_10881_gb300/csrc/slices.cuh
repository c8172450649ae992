// slices.cuh -- series coefficients as exact integer slices for the tensor cores.
//
// A coefficient on grid g is L balanced B-bit digits, digit p weighing
// 2^(B (g - 1 - p)) (the form of digits.cuh); every digit is held as two slices of
// W = B / 2 bits, digit = s_0 2^W + s_1, both within 2^(W-1) in magnitude.  A slice
// is one f16 number in units of 2^-24, the format's smallest subnormal: integers up
// to 1024 in magnitude are exact there, and their bits are the magnitude itself with
// the sign in bit 15.  One 32-bit word holds one digit, s_0 in its upper half.
//
// Products of two slices are at most 2^(2W-2); an fp32 accumulator of the f16 mma
// takes 2^24 of them exactly (checked on this GPU against integer sums, subnormal
// operands included), and its upper part is moved into a second fp32 number before
// that.  W is 9 or 10 bits: f16 would hold 11, but each further bit leaves a quarter
// of the products per move.  Two slices fill a word, so a shift by whole digits (two
// coefficients on different grids) is a shift by whole words.
//
// e4m3 slices of 5 bits were measured first: four times the products, and the e4m3
// mma.sync runs at the f16 form's multiply-add rate on this GPU, behind conversions
// of its operands (2.4 times slower than the integer pipe).
#pragma once
#include "digits.cuh"

namespace pes {

// Bits of a slice: 10 where that saves a 16-slice block of a coefficient (k = 10: 58
// slices instead of 66), else 9.
PES_HDC int slice_bits(int k) { return k >= 10 ? 10 : 9; }
PES_HDC int slice_digit_bits(int k) { return 2 * slice_bits(k); }

// Digits per coefficient: at least as many bits below the top digit as the
// 28-bit digits of the same k keep (digits_for_k), so at least 53 k + 28.
PES_HDC int slice_digits(int k) {
  return (DIGIT_BITS_INT * (digits_for_k(k, DIGIT_BITS_INT) - 1) + slice_digit_bits(k) - 1) / slice_digit_bits(k) + 1;
}

// Grids below are taken for zero: the line of the 28-bit digits, 2^-2800000.
PES_HDC int32_t slice_grid_low(int k) { return -(-GRID_LOW * DIGIT_BITS_INT / slice_digit_bits(k)); }

// word of a balanced digit v, |v| <= 2^(2W-1)
template <int W>
PES_HD uint32_t slice_encode(int32_t v) {
  constexpr int32_t H = 1 << (W - 1);
  const int32_t hi = (v + H) >> W;
  const int32_t lo = v - hi * (1 << W);
  const uint32_t a = static_cast<uint32_t>(hi < 0 ? 0x8000 - hi : hi);
  const uint32_t b = static_cast<uint32_t>(lo < 0 ? 0x8000 - lo : lo);
  return (a << 16) | b;
}

template <int W>
PES_HD int32_t slice_decode(uint32_t w) {
  const int32_t a = static_cast<int32_t>((w >> 16) & 0x7fffu), b = static_cast<int32_t>(w & 0x7fffu);
  const int32_t lo = (w & 0x8000u) ? -b : b;
  const int32_t hi = (w & 0x80000000u) ? -a : a;
  return hi * (1 << W) + lo;
}

// s_0 2^16 + s_1
PES_HD int32_t slice_halves(uint32_t w) {
  const uint32_t n = (w >> 15) & 0x00010001u;  // signs
  return static_cast<int32_t>(((w & 0x7fff7fffu) ^ (n * 0xffffu)) + n - (n << 16));
}

PES_HD int32_t slice_square(uint32_t w) {
  const int32_t a = static_cast<int32_t>((w >> 16) & 0x7fffu), b = static_cast<int32_t>(w & 0x7fffu);
  return a * a + b * b;
}

// What the workspace keeps of a coefficient beside its digits: the grid in the upper 24
// bits, and in the lower 8 a bound on the sum of its squared slices, one unit per eighth
// of a power of two (0 for a zero coefficient).
PES_HD int32_t slice_meta(int32_t grid, int32_t squares) {
  constexpr int32_t G = 1 << 22;
  if (grid < -G) grid = -G;
  if (grid > G) grid = G;
  const float f = static_cast<float>(squares);
#if defined(__CUDA_ARCH__)
  const int32_t bits = __float_as_int(f);
#else
  int32_t bits;
  std::memcpy(&bits, &f, sizeof(bits));
#endif
  const int32_t q = squares == 0 ? 0 : (bits >> 20) + 1 - (127 << 3);
  return grid * 256 + q;
}
PES_HD int32_t meta_grid(int32_t meta) { return meta >> 8; }
// the bound that q stands for
PES_HD float meta_norm(int32_t q) {
  const int32_t bits = (q + (127 << 3)) << 20;
#if defined(__CUDA_ARCH__)
  return __int_as_float(bits);
#else
  float f;
  std::memcpy(&f, &bits, sizeof(f));
  return f;
#endif
}

// ---------------------------------------------------------------------------
// The sums of the addition stage.  Contributions are added digit by digit (B
// bits); the grids and digit sums that ranks exchange (pes_partial_*) are in
// 28-bit digits, L28 = digits_for_k(k, 28) of them.  Both see the same number: the
// grid G of a sum whose largest contribution lies on grid g has B g - 28 G in
// [B - 28, 16], and the bits of every contribution below the last 28-bit digit are
// dropped (toward zero, digit by digit), in either form: less than one unit of that digit
// a contribution, 2^-(53 k + 28) of the largest (a sum of 28-bit digits drops half a unit
// of it; the products before drop less here than there).
// ---------------------------------------------------------------------------
template <int B>
PES_HD int32_t sum_grid28(int32_t g) {
  return floordiv(B * g + 11, 28);
}
// the largest grid g with that G
template <int B>
PES_HD int32_t sum_anchor(int32_t G) {
  return floordiv(28 * G + 16, B);
}
// B-bit words a sum can hold above its floor
PES_HDC int sum_words(int k) {
  return (DIGIT_BITS_INT * digits_for_k(k, DIGIT_BITS_INT) + 16) / slice_digit_bits(k) + 1;
}
// the digit d of a contribution without its f lowest bits
PES_HD int32_t sum_cut(int32_t d, int f) { return d < 0 ? -((-d >> f) << f) : (d >> f) << f; }

}  // namespace pes
