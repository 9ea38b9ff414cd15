// Which kernel a global product takes (global.cu). Plain arithmetic that also compiles without CUDA, so that the rule can
// be held against its measurements on the host.
#pragma once

#include <stdint.h>

namespace mka {

// Stored values (0: FP64, 1: FP32, 2: BF16), FP64 or FP32 vectors, k of them, n atoms, nnzb blocks; wide: the kernel by
// slots would use eight of them. True: a thread per row (spmv_rows_kernel).
//
// The kernel by slots takes 8 (wide: 16) blocks of a row at a time and reads four atoms ahead, which pays where rows
// fill its steps: with 13 blocks a row it is the faster one except for much memory. A thread per row has no idle lanes on
// short rows, and half the instructions a byte of FP64 values, whose loads are the widest. Microseconds by slots / by rows:
//   one block a row: 262,144 atoms, FP64 values and vectors, k = 2, 145 / 28; FP32, k = 4, 34 / 13; 512 atoms, FP64, k = 1,
//   5.9 / 4.5
//   4.4 blocks: 262,144 atoms, FP64, k = 4, 233 / 183; BF16 values, FP32 vectors, k = 4, 39 / 31; 32,768 atoms, FP32, k = 4,
//   8.2 / 6.8
//   8 and 16 blocks, where some rows need one more step: 262,144 atoms, FP64, k = 1, 137 / 93 and 194 / 147
//   12 blocks: 262,144 atoms, FP64, k = 1, 133 / 119, k = 4, 436 / 445; FP32, k = 1, 39 / 51; 8,000 atoms, FP64, k = 1, 8.4 / 10
constexpr bool spmv_by_rows(int values, bool x64, int k, int64_t n, int64_t nnzb, bool wide) {
  const double m = (double)nnzb / (double)n;
  if (m < 1.5) {
    if (values == 0 || (x64 && k == 1)) return true;
    return n >= (x64 && k == 2 ? 1500 : 6000);
  }
  if (values == 0) {
    if (x64 && k == 4) return n >= 524288 || (m < 2.5 && n >= 24000) || (m > 3.5 && m < 5.5 && n >= 6000);
    if (n >= 65536) return true;
    if (!x64 && k == 4) return n >= 24000 && m < 5.0;
    if (!x64 && k == 2) return n >= 24000 || (n >= 6000 && m < 5.0);
    const int step = wide ? 16 : 8, steps = (int)((m + 1.5) / step) + 1;   // of most rows, which differ by a few blocks
    return n >= 6000 && (m > 20.0 || m < 0.7 * step * steps);
  }
  if (x64) return k == 4 && m < 2.5 && n >= 65536;
  if (n < 24000) return false;
  if (values == 1) return m < 5.0 && (k > 1 || n < 131072 || m < 2.5);
  return k == 1 || m < 5.0 || (k == 2 && n >= 131072) || (k == 4 && n >= 65536 && m < 10.0);
}

}  // namespace mka
