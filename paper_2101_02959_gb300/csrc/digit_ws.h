// Sizes and layout of the workspace of the digit products (digits.cu): host arithmetic only, shared by
// the code that allocates it and the code that launches into it.
#pragma once
#include <algorithm>
#include <cstddef>

namespace bd {

constexpr int kPanel64 = 64;   // panel width where the panels too are solved on the tensor cores
constexpr int kPanelExp = 72;  // ints per matrix for the column exponents of a panel solve, and a flag
constexpr int kUpdM = 128;     // rows of an update's tile
constexpr int kUpdN = 64;      // its columns
constexpr int kUpdK = 32;      // columns of K per digit block (one 64-byte row of bf16)
constexpr int kDigitBlk = 64 * kUpdK * 2;  // bytes of one digit plane of 64 rows x kUpdK columns
constexpr int kSliceK = 1024;  // columns whose digit planes the workspace holds at a time

// digits of an entry and columns of a scaling group
template <typename T> struct DigitDims;
template <> struct DigitDims<double> { static constexpr int D = 7, Grp = 128; };
template <> struct DigitDims<float> { static constexpr int D = 3, Grp = 64; };
static_assert(kPanel64 <= DigitDims<double>::Grp && kPanel64 <= DigitDims<float>::Grp,
              "a panel inverse is one scaling group");

inline int digit_ceil(int a, int b) { return (a + b - 1) / b; }
inline int digit_rows(int rows) { return digit_ceil(std::max(rows, 1), kUpdM) * kUpdM; }
template <typename T>
size_t digit_planes(int rows, int cols) {
  return (size_t)digit_ceil(cols, kUpdK) * DigitDims<T>::D * digit_ceil(rows, 64) * kDigitBlk;
}
// one operand of `rows` rows and `cols` columns: planes, and the row exponents of its groups
template <typename T>
size_t digit_operand(int rows, int cols) {
  const int r = digit_rows(rows);
  return digit_planes<T>(r, cols) + (size_t)digit_ceil(cols, DigitDims<T>::Grp) * r * sizeof(int);
}

// Byte offsets of an update of `count` matrices, `cols` columns of K at a time: the planes of the rows
// at 0, those of the panel inverses, then both sets of exponents.
struct UpdLayout {
  size_t inv, ex, ex_inv, bytes;
};
template <typename T>
UpdLayout upd_layout(int count, int rows, int cols) {
  const size_t n = (size_t)std::max(count, 1);
  const int r = digit_rows(rows);
  UpdLayout l;
  l.inv = n * digit_planes<T>(r, cols);
  l.ex = l.inv + n * digit_planes<T>(kUpdN, kPanel64);
  l.ex_inv = l.ex + n * (size_t)digit_ceil(cols, DigitDims<T>::Grp) * r * sizeof(int);
  l.bytes = l.ex_inv + n * kUpdN * sizeof(int);
  return l;
}

// Workspace of `count` matrices of max_rows rows and max_e eliminated columns.  A panel is laid out at
// its full width whatever max_e is.
template <typename T>
size_t slice_bytes(int count, int max_rows, int max_e) {
  return upd_layout<T>(count, max_rows, std::min(std::max(max_e, kPanel64), kSliceK)).bytes;
}
// Workspace of `count` products of matrices of order max_n.
template <typename T>
size_t product_bytes(int count, int max_n) {
  return 2 * (size_t)std::max(count, 1) * digit_operand<T>(max_n, std::max(max_n, 1));
}
// Matrices of a run: as many of `count` as the workspace holds; 0 when it does not hold one.
inline int digit_run(size_t ws_bytes, size_t one, int count) {
  return (int)std::min<size_t>((size_t)count, ws_bytes / one);
}

}  // namespace bd
