// The places of the nonzero coefficients of Strassen's algorithm, nested once (FMM_LEVELS 2, the default) or plain (1), for
// kernels whose lists are compiled in: encode_pattern.cu and decode_pattern.cu are compiled once for each.  Internal linkage.
#pragma once
#ifndef FMM_LEVELS
#define FMM_LEVELS 2
#endif
#if FMM_LEVELS == 2
#define FMM_PATTERN(name) name##_two_level
#else
#define FMM_PATTERN(name) name##_one_level
#endif
#include <type_traits>
#include <utility>

namespace {

constexpr int kLevels = FMM_LEVELS, kProducts = kLevels == 2 ? 49 : 7, kGrid = 2 * kLevels, kCells = kGrid * kGrid;

// nonzero places of the one-level algorithm's coefficients, as (row, column) bits 2 * row + column of U (A), V (B), W (C)
constexpr unsigned char kU[7] = {0b1001, 0b1100, 0b0001, 0b1000, 0b0011, 0b0101, 0b1010};
constexpr unsigned char kV[7] = {0b1001, 0b0001, 0b1010, 0b0101, 0b1000, 0b0011, 0b1100};
constexpr unsigned char kW[7] = {0b1001, 0b1100, 0b1010, 0b0101, 0b0011, 0b1000, 0b0001};

// those of them that are -1 in the built-in algorithm; the others are 1
constexpr unsigned char kUMinus[7] = {0, 0, 0, 0, 0, 0b0001, 0b1000};
constexpr unsigned char kVMinus[7] = {0, 0, 0b1000, 0b0001, 0, 0, 0};

struct Pattern {
  int off[kProducts + 1] = {};
  unsigned char cell[kProducts * kCells] = {};
  signed char sign[kProducts * kCells] = {};      // of the built-in algorithm's coefficient, of its inner factor where the outer one is
                                                  // dense (encode patterns)
};
// entries with dense coefficients of the outermost level: dense (x) S has 4 * 7 * 12 where S (x) S has 144, dense 28 where S has 12
constexpr int kMaxEntries = kLevels == 2 ? 336 : 28;
// is coefficient (x, y) of product r nonzero, where nz are the patterns of one level
constexpr bool is_entry(const unsigned char (&nz)[7], int r, int x, int y, bool dense) {
  const int outer = kLevels == 2 ? x / 2 * 2 + y / 2 : x * 2 + y, inner = x % 2 * 2 + y % 2;
  return (dense || ((nz[kLevels == 2 ? r / 7 : r] >> outer) & 1)) && (kLevels == 1 || ((nz[r % 7] >> inner) & 1));
}

// f(integral_constant) for every index of the sequence
template <int... i, typename F>
__device__ __forceinline__ void for_each(std::integer_sequence<int, i...>, F&& f) { (f(std::integral_constant<int, i>{}), ...); }

}  // namespace
