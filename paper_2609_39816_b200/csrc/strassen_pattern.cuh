// The places of the nonzero coefficients of two-level Strassen, for kernels whose lists are compiled in.  Internal linkage.
#pragma once
#include <type_traits>
#include <utility>

namespace {

constexpr int kProducts = 49, kCells = 16;

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
constexpr int kMaxEntries = 336;      // dense (x) S: 4 * 7 * 12; S (x) S has 144

// f(integral_constant) for every index of the sequence
template <int... i, typename F>
__device__ __forceinline__ void for_each(std::integer_sequence<int, i...>, F&& f) { (f(std::integral_constant<int, i>{}), ...); }

}  // namespace
