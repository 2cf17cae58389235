// Orientation of a batched product on 128-row tensor-core tiles (host).
#pragma once
#include <algorithm>

namespace mpslcc {

// How C_b = A_b B_b^T (m x n, b < nb, C_b at b sC with rows ldc apart; A or B
// may be shared by all entries) becomes one product D = X Y^T with X on the
// tile's 128-row side and Y on its column side: D(r, j) of entry e lies at
// (r / rpb) bstride + (r % rpb) ldr + j cst + e cbatch.
struct TcFold {
  bool swap;                // X = B, Y = A (else X = A, Y = B)
  int rows, cols, batch;    // rows of X and of Y, entries left
  int rpb;
  long long bstride;
  int ldr, cst;
  long long cbatch;
};

// An operand of its own per entry beside a shared one is a stack of nb times
// its rows: put on the row side it needs no batch at all.  Boxes of the fused
// operators have one or two rows against some 20 x 80 such rows; entry by
// entry they filled 0.1 % of their tiles (185788 tiles and 4.5 ms for the
// operators of a BF16x6 right-hand side; 0.24 ms with the stacks on the row
// side).  Between the two orientations the
// one that moves fewer operand rows through the tiles is taken; on a tie the
// swapped one, whose stores run along C's rows.
inline TcFold tc_fold(int m, int n, int nb, bool a3, bool b3, int ldc, long long sC, int cap) {
  TcFold f[2];
  long long cost[2];
  for (int s = 0; s < 2; ++s) {
    const bool own = s ? b3 : a3, other = s ? a3 : b3;   // X, Y have an entry each
    const bool fold = nb > 1 && own && !other && (long long)nb * (s ? n : m) < (1LL << 30);
    TcFold& t = f[s];
    t.swap = s == 1;
    t.rows = (s ? n : m) * (fold ? nb : 1);
    t.cols = s ? m : n;
    t.batch = fold ? 1 : nb;
    t.rpb = fold ? (s ? n : m) : 1 << 30;
    t.bstride = fold ? sC : 0;
    t.ldr = s ? 1 : ldc;
    t.cst = s ? ldc : 1;
    t.cbatch = fold ? 0 : sC;
    const int nt = std::min(cap, (t.cols + 15) / 16 * 16);
    cost[s] = (long long)t.batch * ((t.rows + 127) / 128) * ((t.cols + nt - 1) / nt) * (128 + nt);
  }
  return cost[1] <= cost[0] ? f[1] : f[0];
}

}  // namespace mpslcc
