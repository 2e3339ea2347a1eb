// Host side of the split products' sine tables (modes_split.cu): the digits of a
// table value, the scales of the rows, and what the digits say about the sums.
// Plain C++.
#pragma once

#include <algorithm>
#include <cmath>
#include <cstdint>

#ifdef __CUDACC__
#define PP_HOST_DEVICE __host__ __device__
#else
#define PP_HOST_DEVICE
#endif

namespace pp {

// Digits of a split value, and products kept per pair of split values.
constexpr int kSplitDigits = 6;
constexpr int kSplitBits = 9;

// Biased values: X + kSplitBias has the non-negative 9-bit fields d_i + 256
// (i = 5 .. 1) and d_0 + 512 above them
constexpr long long kSplitBiasLow = 256LL * (1 + (1LL << 9) + (1LL << 18) + (1LL << 27) + (1LL << 36));
constexpr long long kSplitBias = kSplitBiasLow + (512LL << 45);
PP_HOST_DEVICE inline int split_digit(long long X, int digit) {
  X += kSplitBias;
  return digit == 0 ? int(X >> 45) - 512 : int((X >> (kSplitBits * (kSplitDigits - 1 - digit))) & 511) - 256;
}

// A table row's scale: its digits are those of the row times 2^s, 0 <= s <=
// kMaxRowScale, or kZeroRow where the row is zero; stored as s 2^20 (an FP64
// number's exponent is there in its high word), for rows padded to a multiple of 16
constexpr int kMaxRowScale = 64, kZeroRow = 2047;
// row r's place: 16 rows are kept as a lane's four, 2t, 2t + 1, 2t + 8, 2t + 9, for t = 0 .. 3
PP_HOST_DEVICE inline int scale_index(int r) {
  return r / 16 * 16 + (r % 8) / 2 * 4 + (r % 16) / 8 * 2 + r % 2;
}
inline int split_padded(int rows) { return (rows + 15) / 16 * 16; }
struct RowScale {
  const int* rows;
  int plain0, plain1;        // 16-row steps of the table in which every scale is 0
};

// the powers of two that bring each row's largest value into [1/2, 1] (.rows is left null)
inline RowScale table_scales(const double* tab, int rows, int slots, int* scale) {
  for (int r = 0; r < split_padded(rows); ++r) {
    double top = 0.0;
    for (int k = 0; r < rows && k < slots; ++k) top = std::fmax(top, std::fabs(tab[size_t(r) * slots + k]));
    int e = 0;
    if (top > 0.0) std::frexp(top, &e);
    const int s = top > 0.0 ? std::min(std::max(-e, 0), kMaxRowScale) : kZeroRow;
    scale[scale_index(r)] = s * (1 << 20);
  }
  RowScale out{nullptr, 0, 0};                       // the longest run of steps without a scale
  for (int k = 0, from = 0; k < split_padded(rows) / 16; ++k) {
    for (int r = 16 * k; r < 16 * k + 16 && r < rows; ++r)
      if (scale[scale_index(r)] != 0) from = k + 1;
    if (k + 1 - from > out.plain1 - out.plain0) {
      out.plain0 = from;
      out.plain1 = k + 1;
    }
  }
  return out;
}

// |digits| of the table value (r, k), scaled
inline void table_digits(const double* tab, const int* scale, int slots, int r, int k, long (&d)[kSplitDigits]) {
  const int s = std::min(scale[scale_index(r)] >> 20, kMaxRowScale);
  const long long X = std::llrint(std::ldexp(tab[size_t(r) * slots + k], 53 + s));
  for (int j = 0; j < kSplitDigits; ++j) d[j] = std::labs(long(split_digit(X, j)));
}
// the largest |sum over i + j = w of d_i t_j| where the |t_j| add up to sum[j] and |d_i| <= 256, |d_0| <= first
inline long weight_bound(const long (&sum)[kSplitDigits], int w, long first) {
  long bound = 0;
  for (int j = 0; j <= w; ++j) bound += sum[j] * (j == w ? first : 256L);
  return bound;
}

// the expansion over this table [rows][slots] can take its sums off the
// accumulators' bits: every weight's sum stays below 2^22 (|d_0| <= 1024 there)
inline bool expand_sums_small(const double* tab, const int* scale, int rows, int slots, bool halves) {
  const int kh = halves ? slots / 2 : slots;
  if (kh > 16) return false;
  for (int r = 0; r < rows; ++r)
    for (int h = 0; h < (halves ? 2 : 1); ++h) {
      long sum[kSplitDigits] = {}, d[kSplitDigits];
      for (int k = 0; k < kh; ++k) {
        table_digits(tab, scale, slots, r, h * kh + k, d);
        for (int j = 0; j < kSplitDigits; ++j) sum[j] += d[j];
      }
      for (int w = 0; w < kSplitDigits; ++w)
        if (weight_bound(sum, w, 1024) >= 1L << 22) return false;
    }
  return true;
}

// 16-row steps, 4, 2 or 1, that a contraction over this table may sum in one set
// of accumulators: the sums of the weights 0 .. 4 then stay within 2^24 for every
// data (halves: mirror pairs, whose leading digits go to 512).  One step always
// does: 16 (512 + 4 256) 256 < 2^24.
inline int contract_steps(const double* tab, const int* scale, int rows, int slots, bool halves) {
  int steps = 4;
  for (int k = 0; k < slots; ++k)
    for (int r0 = 0; r0 < rows; r0 += 16 * steps) {
      long sum[kSplitDigits] = {}, d[kSplitDigits];
      for (int r = r0; r < std::min(rows, r0 + 16 * steps); ++r) {
        table_digits(tab, scale, slots, r, k, d);
        for (int j = 0; j < kSplitDigits; ++j) sum[j] += d[j];
      }
      bool fits = true;
      for (int w = 0; w < kSplitDigits - 1; ++w) fits = fits && weight_bound(sum, w, halves ? 512 : 256) <= 1L << 24;
      if (!fits && steps > 1) {
        steps /= 2;
        k = -1;                                      // from the start with shorter runs
        break;
      }
    }
  return steps;
}

}  // namespace pp
