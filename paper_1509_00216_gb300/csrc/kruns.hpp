// K runs of the sigma tasks (host side): the column ranges of an operand that
// hold a task's non-zero local pieces, merged into the runs a kernel reads.
// Header-only and free of CUDA, so that the host logic is tested on its own.
#pragma once
#include <algorithm>
#include <utility>
#include <vector>

namespace mpslcc {

// One run of a tensor-core task: `steps` K steps of KT columns from column kx.
struct KRun {
  long kx, steps;
};

// Runs of a tensor-core task whose non-zero columns come as ranges [a, b) of
// the operands' K extent (any order; empty ranges are dropped).  Each run
// starts on an 8-element boundary (a 16-byte TMA coordinate for 16-bit types)
// and is read in whole steps of KT columns.  A range that starts (rounded
// down to 8) before the open run's last step ends joins that run, so no
// column is read by two runs; the columns a run reads outside the ranges must
// be zero in one operand, so that they add nothing.
struct RunBuilder {   // the ranges one by one, in ascending order
  int KT;
  std::vector<KRun> runs;
  long de = 0;        // end of the data the open run must cover
  explicit RunBuilder(int KT_) : KT(KT_) {}
  void add(long a, long b) {
    if (b <= a) return;
    const long a8 = a & ~7L;
    if (!runs.empty() && a8 < runs.back().kx + runs.back().steps * KT) {
      de = std::max(de, b);
      runs.back().steps = (de - runs.back().kx + KT - 1) / KT;
    } else {
      runs.push_back({a8, (b - a8 + KT - 1) / KT});
      de = b;
    }
  }
};

// The ranges in any order (the products add theirs in ascending order).
inline std::vector<KRun> merge_runs(std::vector<std::pair<long, long>>& r, int KT) {
  std::sort(r.begin(), r.end());
  RunBuilder out(KT);
  for (const auto& x : r) out.add(x.first, x.second);
  return std::move(out.runs);
}

// The same ranges merged exactly (sorted, disjoint, neither overlapping nor
// touching), for kernels that read element by element (the FP64 path).
inline std::vector<std::pair<long, long>> merge_exact(std::vector<std::pair<long, long>>& r) {
  if (!std::is_sorted(r.begin(), r.end())) std::sort(r.begin(), r.end());
  std::vector<std::pair<long, long>> m;
  for (const auto& x : r) {
    if (x.second <= x.first) continue;
    if (!m.empty() && x.first <= m.back().second) m.back().second = std::max(m.back().second, x.second);
    else m.push_back(x);
  }
  return m;
}

}  // namespace mpslcc
