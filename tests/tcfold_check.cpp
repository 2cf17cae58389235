// Orientation of batched products (tcfold.hpp): whatever is chosen, element
// (i, j) of entry b must land at b sC + i ldc + j, from the rows of the
// operands that belong to it.  Exits 0 when every case holds.
#include <cstdio>
#include <random>

#include "tcfold.hpp"

int main() {
  std::mt19937_64 rng(7);
  int folded = 0, swapped = 0;
  for (int trial = 0; trial < 4000; ++trial) {
    auto pick = [&](int hi) { return 1 + (int)(rng() % (trial % 3 ? hi : 3)); };
    const int m = pick(150), n = pick(300), nb = pick(20);
    const bool a3 = nb > 1 && rng() % 2, b3 = nb > 1 && rng() % 2;
    const int ldc = n + (int)(rng() % 5);
    const long long sC = rng() % 2 ? (long long)m * ldc : n + (long long)(rng() % 1000);
    const auto f = mpslcc::tc_fold(m, n, nb, a3, b3, ldc, sC, rng() % 2 ? 64 : 256);
    const bool fold = f.batch == 1 && nb > 1;
    folded += fold;
    swapped += f.swap;
    if ((long long)f.rows * f.cols * f.batch != (long long)m * n * nb) return std::printf("FAIL size %d\n", trial), 1;
    if (fold && ((f.swap ? a3 : b3) || !(f.swap ? b3 : a3))) return std::printf("FAIL fold %d\n", trial), 1;
    for (int s = 0; s < 200; ++s) {
      const int i = (int)(rng() % m), j = (int)(rng() % n), b = (int)(rng() % nb);
      const int x = f.swap ? j : i, y = f.swap ? i : j;     // row of the entry's X and Y
      const int r = fold ? b * (f.swap ? n : m) + x : x, e = fold ? 0 : b;
      const long long at = (long long)(r / f.rpb) * f.bstride + (long long)(r % f.rpb) * f.ldr + (long long)y * f.cst +
                           e * f.cbatch;
      if (r >= f.rows || y >= f.cols || at != b * sC + (long long)i * ldc + j)
        return std::printf("FAIL address %d\n", trial), 1;
    }
  }
  if (folded < 100 || swapped < 100) return std::printf("FAIL coverage\n"), 1;
  std::printf("ok\n");
  return 0;
}
