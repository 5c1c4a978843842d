// FP64-accurate complex contractions on the tensor cores by exact integer slices (the error-free splitting of Ozaki,
// Ogita, Oishi and Rump, Numer. Algorithms 59 (2012), in fixed point).
//
// A real x with |x| < S = 2^s becomes the integer v = round(x 2^52 / S) and six balanced digits of nine bits,
// v = sum_i d_i 512^(5-i), d_i in [-256, 255], |d_0| <= 129.  Each digit is exact in FP16; the product of two digit
// matrices over K <= 24 and the sum of the up to six products with i + j = s are integers below 2^23, so
// mma.sync (FP16 operands, FP32 accumulators) forms them exactly: D_s = sum_{i+j=s} A_i B_j.  The levels s = 0..6 are
// added up in 64-bit integers, sum_s D_s 512^(10-s) / 2^52.  The dropped levels are at most 0.09 of the last place with six
// branches and 0.19 with twelve (every digit at the end of its range), 0.005 and 0.007 rms.  The result is the product to
// about 2^-53 of the scale, the rounding that FP64 has for its largest elements.
//
// A complex product over nb components is a real one over K = 2 nb: row elements (re, im) at K = 2 l, 2 l + 1, and
// two columns (re, im) per output.  FP64 runs at 2 lane FMAs per clock and SM on this chip, mma.sync at about 950
// FP16 multiply-adds: the 26 digit products cost 2.7k clocks per 216 x 12 x 12 contraction pair against 20k.
#pragma once
#include <cuda_fp16.h>

#include "fp_internal.cuh"

namespace fp {
namespace slices {

// What a fixed scale costs, and how a caller bounds it.  The error of a result is about 2^-53 S (a few units at worst),
// S the scale of its block, however small the result is.  FP64 loses less where the block's large elements meet zeros of
// the other operands: force constants that differ by orders of magnitude between sublattices, modes confined to one.  So
// the sums keep account: a result below kWeak S counts as weak, and beside a sum of |W|^2 g the S^2 g of its weak terms are
// bounded by their number and the largest.  The others are exact to about 2^-53 / kWeak = 5e-13 at worst; the weak ones
// together change the sum by less than that where the bound stays below kWeak^-2 = 2^24 of it.  A sum that fails this is
// evaluated without slices.  On the crystals of the tests the bound is 2^0 to 2^8 of the sum at 300 K, 2^20 at most at 10 K.
// The account costs 0.2 % of the time with one temperature on diamond 6x6x6 (119.5 -> 119.8 ms), 0.8 % with three on LiCoO2
// 4x3x3 (20.2 -> 20.4), 2.5 % with eight on diamond 5x5x5 (33.1 -> 33.9).
constexpr int kWeakExponent = -12;              // kWeak = 2^-12
constexpr double kWeakLimit = 1.0 / 16777216.0;  // kWeak^2

constexpr int kDigits = 6;
constexpr int kLevels = 7;
constexpr unsigned long long kDigitBias = 256ull * (1ull + 512ull + (1ull << 18) + (1ull << 27) + (1ull << 36) + (1ull << 45));

// shapes for nb = 6 or 12 branches
template <int NB>
struct Shape {
  static constexpr int kTiles = NB == 6 ? 2 : 3;   // column tiles of 8: nb = 6 puts the last four reals one per lane
  static constexpr int kA = NB == 6 ? 4 : 6;       // A registers per digit and row tile (K = 16, or 16 + 8)
  static constexpr int kB = NB == 6 ? 2 : 3;       // B registers per digit and column tile
  static constexpr int kRow = NB == 6 ? 36 : 76;   // words per row of digits (six digits x nb words; padded against
                                                   // bank conflicts)
  static constexpr int kOperand = kDigits * kTiles * 32 * kB;  // words of one B operand in fragment order
};

// digit i of the biased value v (v + kDigitBias) of two reals as FP16 integers: (re, im) in (low, high) half
__device__ __forceinline__ unsigned pack_digit(int i, unsigned long long re, unsigned long long im) {
  const unsigned rl = (unsigned)re, rh = (unsigned)(re >> 32), il = (unsigned)im, ih = (unsigned)(im >> 32);
  unsigned r, m;  // the nine bits of re at bit 0, those of im at bit 16
  switch (i) {
    case 5: r = rl; m = il << 16; break;
    case 4: r = rl >> 9; m = il << 7; break;
    case 3: r = rl >> 18; m = il >> 2; break;
    case 2: r = __funnelshift_r(rl, rh, 27); m = __funnelshift_r(il, ih, 11); break;
    case 1: r = rh >> 4; m = ih << 12; break;
    default: r = rh >> 13; m = ih << 3; break;
  }
  // 0x6400 + n is the FP16 number 1024 + n; subtracting 1280 leaves n - 256 exactly
  const unsigned w = (r & 0x1ffu) | 0x64006400u | (m & 0x1ff0000u);
  const __half2 h = __hsub2(*reinterpret_cast<const __half2*>(&w), __half2half2(__ushort_as_half(0x6500)));
  return *reinterpret_cast<const unsigned*>(&h);
}

// biased fixed-point value of x for the scale 2^s, |x| < 2^s (rounded to nearest, ties away from zero)
__device__ __forceinline__ unsigned long long fixed_from(double x, int s) {
  const long long b = __double_as_longlong(x);
  const int sh = max(min(1023 + s - (int)((b >> 52) & 0x7ff), 60), 1);
  const unsigned long long m = ((unsigned long long)b & 0xfffffffffffffull) | 0x10000000000000ull;
  const unsigned long long v = ((m >> (sh - 1)) + 1ull) >> 1;
  const long long sign = b >> 63;
  return (unsigned long long)(((long long)v ^ sign) - sign) + kDigitBias;
}

// Level sums of one element as integers plus kLB: float + 1.5 2^23 holds an integer below 2^22 in its low bits.  With
// twelve branches (K = 24) levels 3 and 4 can reach 2^22.6 and are converted (no bias).  Levels 5 and 6 count for 2^-7
// and 2^-16 (2^-8 and 2^-17 in combine_magic): their sum is rounded to that place at once.
constexpr long long kLB = 0x4B400000ll;
template <int NB>
__device__ __forceinline__ int level_bits(int s, float d) {
  if (NB == 12 && s >= 3) return __float2int_rn(d);
  return __float_as_int(__fadd_rn(d, 12582912.f));
}
template <int NB>
__host__ __device__ constexpr unsigned long long level_bias(unsigned long long w5, unsigned long long w4, unsigned long long w3,
                                                            unsigned long long w2, unsigned long long w1, unsigned long long w0) {
  return (unsigned long long)kLB * (w5 + (NB == 12 ? 0ull : w4 + w3) + w2 + w1 + w0);
}

// sum_s D_s 2^(38 - 9 s) + kDigitBias: the product of two fixed-point operands (2^52 = 1) in the same fixed point
template <int NB>
__device__ __forceinline__ unsigned long long combine_fixed(const float D[kLevels]) {
  const int q = __float_as_int(__fmaf_rn(__fmaf_rn(D[6], 1.f / 512.f, D[5]), 1.f / 128.f, 12582912.f));
  long long acc = (long long)q + (long long)level_bits<NB>(4, D[4]) * 4ll;
  acc += (long long)level_bits<NB>(3, D[3]) * 2048ll;
  acc += (long long)level_bits<NB>(2, D[2]) * 1048576ll;
  acc += (long long)level_bits<NB>(1, D[1]) * 536870912ll;
  constexpr unsigned long long bias = level_bias<NB>(1ull, 4ull, 2048ull, 1048576ull, 536870912ull, 1ull << 38);
  return (unsigned long long)acc + ((unsigned long long)((unsigned)level_bits<NB>(0, D[0]) << 6) << 32) + (kDigitBias - bias);
}

// Half of that value, as the bits of 1.5 2^52 + value: subtracting kMagic as a double leaves the product scaled by 2^51
constexpr double kMagic = 6755399441055744.0;
template <int NB>
__device__ __forceinline__ double combine_magic(const float D[kLevels]) {
  const int q = __float_as_int(__fmaf_rn(__fmaf_rn(D[6], 1.f / 512.f, D[5]), 1.f / 256.f, 12582912.f));
  long long acc = (long long)q + (long long)level_bits<NB>(4, D[4]) * 2ll;
  acc += (long long)level_bits<NB>(3, D[3]) * 1024ll;
  acc += (long long)level_bits<NB>(2, D[2]) * 524288ll;
  acc += (long long)level_bits<NB>(1, D[1]) * 268435456ll;
  constexpr unsigned long long bias = level_bias<NB>(1ull, 2ull, 1024ull, 524288ull, 268435456ull, 1ull << 37);
  constexpr unsigned long long magic = 0x4338000000000000ull;  // kMagic: its last place is 1
  const unsigned long long v =
      (unsigned long long)acc + ((unsigned long long)((unsigned)level_bits<NB>(0, D[0]) << 5) << 32) + (magic - bias);
  return __longlong_as_double((long long)v);
}

__device__ __forceinline__ void mma16(float c[4], const unsigned* a, unsigned b0, unsigned b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3},{%4,%5,%6,%7},{%8,%9},{%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void mma8(float c[4], unsigned a0, unsigned a1, unsigned b0) {
  asm("mma.sync.aligned.m16n8k8.row.col.f32.f16.f16.f32 {%0,%1,%2,%3},{%4,%5},{%6},{%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a0), "r"(a1), "r"(b0));
}

// A fragments (six digits) of the 16 rows from `row0`, from the digit rows in shared memory (kRow words each, word
// i nb + l: digit i of complex l)
template <int NB>
__device__ __forceinline__ void load_a(const unsigned* dig, int row0, int lane, unsigned (*af)[Shape<NB>::kA]) {
  const int g = lane >> 2, t = lane & 3;
  const unsigned *p = dig + (row0 + g) * Shape<NB>::kRow + t, *p8 = p + 8 * Shape<NB>::kRow;
#pragma unroll
  for (int i = 0; i < kDigits; ++i) {
    af[i][0] = p[i * NB];
    af[i][1] = p8[i * NB];
    if constexpr (NB == 6) {
      af[i][2] = t < 2 ? p[i * NB + 4] : 0u;
      af[i][3] = t < 2 ? p8[i * NB + 4] : 0u;
    } else {
      af[i][2] = p[i * NB + 4];
      af[i][3] = p8[i * NB + 4];
      af[i][4] = p[i * NB + 8];
      af[i][5] = p8[i * NB + 8];
    }
  }
}

// level sums of a 16 x 8 tile: acc[s] += sum over i + j = s of A_i B_j
template <int NB>
__device__ __forceinline__ void contract(float (*acc)[4], const unsigned (*af)[Shape<NB>::kA],
                                         const unsigned (*bf)[Shape<NB>::kB]) {
#pragma unroll
  for (int s = 0; s < kLevels; ++s)
#pragma unroll
    for (int c = 0; c < 4; ++c) acc[s][c] = 0.f;
#pragma unroll
  for (int i = 0; i < kDigits; ++i)
#pragma unroll
    for (int j = 0; j < kDigits; ++j)
      if (i + j < kLevels) {
        mma16(acc[i + j], af[i], bf[j][0], bf[j][1]);
        if constexpr (NB == 12) mma8(acc[i + j], af[i][4], af[i][5], bf[j][2]);
      }
}

// B fragments of one column tile, from an operand in fragment order
template <int NB>
__device__ __forceinline__ void load_b(const unsigned* op, int tile, int lane, unsigned (*bf)[Shape<NB>::kB]) {
#pragma unroll
  for (int j = 0; j < kDigits; ++j)
#pragma unroll
    for (int r = 0; r < Shape<NB>::kB; ++r)
      bf[j][r] = op[((j * Shape<NB>::kTiles + tile) * 32 + lane) * Shape<NB>::kB + r];
}

// The two B operands of a grid point in fragment order: 0 contracts with conj(e) (T = A conj(e3)), 1 with e (W = T e2).
// Column n of a tile is real part or imaginary part (ri) of branch j; K = 2 l, 2 l + 1 hold component l.
template <int NB>
__device__ __forceinline__ unsigned operand_word(const double2* ev, int op, int w) {
  const int r = w % Shape<NB>::kB, lane = (w / Shape<NB>::kB) % 32;
  const int tile = (w / (32 * Shape<NB>::kB)) % Shape<NB>::kTiles, dg = w / (32 * Shape<NB>::kB * Shape<NB>::kTiles);
  const int n = lane >> 2, l = (lane & 3) + 4 * r;
  int j, ri;
  bool used = l < NB;
  if (NB == 6 && tile == 1) {
    j = 4 + (n >> 2);
    ri = (n >> 1) & 1;
    used = used && (n & 1) == 0;
  } else {
    j = tile * 4 + (n >> 1);
    ri = n & 1;
  }
  if (!used) return 0u;
  const double2 e = ev[j * NB + l];
  const double x = op == 0 ? (ri ? -e.y : e.x) : (ri ? e.y : e.x);
  const double y = op == 0 ? (ri ? e.x : e.y) : (ri ? e.x : -e.y);
  // components of unit vectors: scale 1 (a component of modulus 1 is 2^52, inside the top digit's range)
  const unsigned long long vx = (unsigned long long)__double2ll_rn(x * 4503599627370496.0) + kDigitBias;
  const unsigned long long vy = (unsigned long long)__double2ll_rn(y * 4503599627370496.0) + kDigitBias;
  unsigned out = 0;
#pragma unroll
  for (int i = 0; i < kDigits; ++i)
    if (i == dg) out = pack_digit(i, vx, vy);
  return out;
}

}  // namespace slices
}  // namespace fp
