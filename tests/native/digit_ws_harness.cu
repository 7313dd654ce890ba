// Host-only harness for the workspace of the digit products (digit_ws.h): reads queries
// "f|d count rows e cols" and prints per query the bytes allocated for (count, rows, e), the run of
// matrices an update of `cols` columns of K takes from it, and that run's layout (offsets, end).
#include <cstdio>

#include "digit_ws.h"

template <typename T>
static void answer(int count, int rows, int e, int cols) {
  const size_t ws = bd::slice_bytes<T>(count, rows, e);
  const int run = bd::digit_run(ws, bd::upd_layout<T>(1, rows, cols).bytes, count);
  const bd::UpdLayout l = bd::upd_layout<T>(run, rows, cols);
  std::printf("%zu %d %zu %zu %zu %zu\n", ws, run, l.inv, l.ex, l.ex_inv, l.bytes);
}

int main() {
  char t;
  int count, rows, e, cols;
  while (std::scanf(" %c %d %d %d %d", &t, &count, &rows, &e, &cols) == 5) {
    if (t == 'd') answer<double>(count, rows, e, cols);
    else answer<float>(count, rows, e, cols);
  }
  return 0;
}
