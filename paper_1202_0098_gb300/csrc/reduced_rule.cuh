// Which form of the reduced problems a call takes (reduced.cu). Plain integer arithmetic that also compiles without
// CUDA, so that the rule can be held against its measurements on the host.
#pragma once

#include <stdint.h>

namespace mka {

enum ReducedForm {
  RF_LANES = 0,   // one lane per column
  RF_FEW = 1,     // a warp per column (four above nu = 64), eigenvalues by bisection
  RF_TEAMS = 2    // teams of lanes (four warps above nu = 64), eigenvalues by QL
};

constexpr int kTeamMinNu = 5;     // the scratch between the three kernels has nu^2 doubles and holds 5 nu
constexpr int kTeamMaxNu = 160;   // the packed triangles fit in shared memory

// Milliseconds on columns whose matrices fill the band like projected Hamiltonians (lane / few / teams):
//   few columns: the chip is not full, and a column's serial chains count. nu = 30: 4 columns 6.7 / 0.8 / 2.1, 2,048
//   9.0 / 2.2 / 2.7; nu = 100: 148 columns 237 / 8.7 / 23. Below nu = 10 the lane is hardly longer than the bisection and
//   QL shorter: nu = 8, 1,024 columns 0.39 / 0.25 / 0.22, 2,048 0.39 / 0.49 / 0.23.
//   many columns: the lanes have no idle ones and fill the chip by themselves, the sooner the smaller nu is: nu = 8, 6,144
//   columns 0.39 / - / 0.36, 8,192 0.39 / - / 0.42; nu = 16, 12,288 1.86 / - / 1.86; nu = 24, 24,576 7.8 / - / 7.1;
//   nu = 30, 40,960 19.8 / - / 18.1; nu = 33, 16,384 14.7 / - / 14.8; nu = 64, 16,384 116 / - / 76. Above nu = 64 one or two
//   columns share an SM: nu = 65, 12,288 116 / 139 / 104, 20,000 133 / - / 165; nu = 100, 12,288 412 / 430 / 360, 20,000
//   462 / - / 588; nu = 128, 10,240 about 850 / - / 785; nu = 160, 8,192 1,611 / 1,518 / 1,446, 20,000 1,847 / - / 3,540.
constexpr ReducedForm reduced_form(int nu, int64_t n_cols) {
  if (nu < kTeamMinNu || nu > kTeamMaxNu) return RF_LANES;
  const int64_t few = nu < 10 ? 768 : 2048;
  const int64_t teams = nu < 8 ? 4096 : nu < 16 ? 6144 : nu < 24 ? 12288 : nu < 28 ? 24576 : nu <= 32 ? 40960
                        : nu <= 64 ? 16384 : nu <= 112 ? 12288 : nu <= 128 ? 10240 : 8192;
  return n_cols <= few ? RF_FEW : n_cols <= teams ? RF_TEAMS : RF_LANES;
}

// The columns a sweep over a system of n atoms picks its form by, whatever its batches are: all of them, so that no batch
// is slower than with a lane per column, or, from nu = 24 to 32, half: up to twice the limit the teams cost 10 % of these
// kernels and save up to half in batches below it (55,296 columns of nu = 30 in batches of 16,384: 27 ms against 38).
constexpr int64_t system_columns(int nu, int64_t n) {
  return 4 * n > 2048 && nu >= 24 && nu <= 32 ? (2 * n > 2048 ? 2 * n : 2049) : 4 * n;
}

}  // namespace mka
