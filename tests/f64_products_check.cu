// FP64 products (gemm_f64.cu) term by term.  `plan` (no GPU): which kernel the
// products below run on.  `run`: every output against the sum taken with error-
// free products and sums, within the error bound of a chain of FP64 fused
// multiply-adds over the same terms.  Exits 0 when every case holds.
#include <cmath>
#include <cstdio>
#include <cstring>
#include <random>
#include <vector>

#include "engine.hpp"

void mpslcc::cuda_check(cudaError_t e, const char* what) {
  if (e != cudaSuccess) throw Error(ST_CUDA, std::string(what) + ": " + cudaGetErrorString(e));
}

using namespace mpslcc;

enum Data { NORMAL, GRADED20, GRADED40, APART, IDENTITY, TINY, POSITIVE, BLOCKS, SPARSE, INFINITE };
enum List { SHORT64, SHORT32, LONG, PIPE };
struct Case {
  const char* name;
  int m, n, k, flags, batch;   // a batch shares B
  Data data;
  List list;
  bool runs;                   // K runs over every other 24 columns
  double alpha, beta;
};

static const Case CASES[] = {
    {"one scaling block, 64 columns", 640, 640, 64, GEMM_TB, 1, NORMAL, SHORT64, false, 1, 0},
    {"graded 2^20", 640, 640, 64, GEMM_TB, 1, GRADED20, SHORT64, false, 1, 0},
    {"graded 2^40", 640, 640, 64, GEMM_TB, 1, GRADED40, SHORT64, false, 1, 0},
    {"graded 2^40, ragged, K along columns", 641, 577, 51, GEMM_TA, 1, GRADED40, SHORT64, false, -0.5, 1},
    {"large against zero", 640, 640, 64, GEMM_TB, 1, APART, SHORT64, false, 1, 0},
    {"unit rows over noise", 640, 600, 100, GEMM_TB, 1, IDENTITY, SHORT64, false, 1, 0},
    {"rows below 2^-959", 640, 640, 64, GEMM_TB, 1, TINY, SHORT64, false, 1, 0},
    {"one sign", 640, 640, 128, GEMM_TB, 1, POSITIVE, SHORT64, false, 1, 0},
    {"sparse", 640, 640, 90, GEMM_TB, 1, SPARSE, SHORT64, false, 1, 0},
    {"sparse, K along columns", 641, 577, 51, GEMM_TA, 1, SPARSE, SHORT64, false, 2, 1},
    {"an infinity", 640, 640, 64, GEMM_TB, 1, INFINITE, SHORT64, false, 1, 0},
    {"32 columns, sparse", 45, 31, 40, 0, 600, SPARSE, SHORT32, false, 1, 0},
    {"32 columns, an infinity", 45, 31, 40, 0, 600, INFINITE, SHORT32, false, 1, 0},
    {"32 columns", 45, 31, 40, GEMM_TB, 600, GRADED40, SHORT32, false, 1, 0},
    {"32 columns, unit rows", 45, 31, 40, 0, 600, IDENTITY, SHORT32, false, 2, 0.5},
    {"32 columns, rows below 2^-959", 45, 31, 40, 0, 600, TINY, SHORT32, false, 1, 0},
    {"several scaling blocks", 300, 200, 2500, GEMM_TB, 1, NORMAL, LONG, false, 1, 0},
    {"several scaling blocks, graded 2^20", 300, 200, 2500, GEMM_TB, 1, GRADED20, LONG, false, 1, 0},
    {"several scaling blocks, graded 2^40, K along columns", 301, 199, 1029, GEMM_TA, 1, GRADED40, LONG, false, 3, 1},
    {"several scaling blocks, large against zero", 300, 200, 2500, 0, 1, APART, LONG, false, 1, 0},
    {"several scaling blocks, rows below 2^-959", 300, 200, 2500, GEMM_TB, 1, TINY, LONG, false, 1, 0},
    {"parts of different magnitude", 300, 200, 1024, GEMM_TB, 1, BLOCKS, LONG, false, 1, 0},
    {"K runs, graded 2^40", 300, 200, 1600, GEMM_TB, 1, GRADED40, LONG, true, 1, 0},
    {"several scaling blocks, sparse", 300, 200, 2500, GEMM_TB, 1, SPARSE, LONG, false, 1, 0},
    {"several scaling blocks, an infinity", 300, 200, 2500, GEMM_TB, 1, INFINITE, LONG, false, 1, 0},
    {"FP64 pipe, graded 2^40", 70, 65, 130, GEMM_TB, 1, GRADED40, PIPE, false, 1, 0},
};

static GemmTask task(const Case& c, const double* A, const double* B, double* C, const int* kr, int nkr, int kv) {
  GemmTask g;
  std::memset(&g, 0, sizeof(g));
  g.A = A; g.B = B; g.C = C;
  g.m = c.m; g.n = c.n; g.k = c.k;
  g.lda = c.flags & GEMM_TA ? c.m : c.k;
  g.ldb = c.flags & GEMM_TB ? c.k : c.n;
  g.ldc = c.n;
  g.batch = c.batch;
  g.sA = (long long)c.m * c.k;
  g.sC = (long long)c.m * c.n;
  g.alpha = c.alpha; g.beta = c.beta;
  g.flags = c.flags;
  g.ksplit = 1;
  if (kr) { g.kr = kr; g.nkr = nkr; g.kv = kv; }
  return g;
}

static std::vector<int> run_table(int k, int& nkr, int& kv) {   // columns [48 r, 48 r + 24)
  std::vector<int> t;
  kv = nkr = 0;
  for (int c = 0; c < k; c += 48, ++nkr) {
    t.push_back(c);
    t.push_back(kv);
    kv += std::min(24, k - c);
  }
  t.push_back(0);
  t.push_back(kv);
  return t;
}

static bool plan_holds(const Case& c, F64Plan& p, const int* kr, int nkr, int kv, const double* A = nullptr,
                       const double* B = nullptr, double* C = nullptr) {
  const GemmTask g = task(c, A, B, C, kr, nkr, kv);
  plan_f64(&g, 1, p);
  const bool ok = c.list == SHORT64   ? p.n[F64_SHORT] == 1 && p.tn == 64
                  : c.list == SHORT32 ? p.n[F64_SHORT] == 1 && p.tn == 32
                  : c.list == LONG    ? p.n[F64_LONG] == 1
                                      : p.n[F64_PIPE] == 1;
  if (!ok)
    printf("%s: lists %d %d %d, %d columns\n", c.name, p.n[F64_SHORT], p.n[F64_LONG], p.n[F64_PIPE], p.tn);
  return ok;
}

// element k of row r of an operand: X (side 0) or Y (side 1)
struct Fill {
  std::mt19937_64 rng;
  std::normal_distribution<double> g;
  double operator()(Data d, int side, int r, int k, int K) {
    const double v = g(rng), f = K > 1 ? (double)k / (K - 1) : 0.0;
    switch (d) {
      case GRADED20: return std::ldexp(v, (int)std::lround((side ? 20 : -20) * f));
      case GRADED40: return std::ldexp(v, (int)std::lround((side ? 40 : -40) * f));
      case APART: return side ? (k % 2 ? v : 0.0) : (k == r % K ? std::ldexp(v, 70) : v);
      case IDENTITY: return side ? v : (k == r % K ? 1.0 : 0x1p-56 * v);
      case TINY: return side || r % 3 ? v : (r % 2 ? v * 1e-295 : v * 4e-320);
      case POSITIVE: return std::fabs(v) + 0.01;
      case BLOCKS: return std::ldexp(v, (k / 100 * 7 + (side ? 3 : 11) * (k / 100)) % 29);
      case SPARSE: return (r * 7 + k * 11 + side) % (side ? 9 : 5) ? 0.0 : std::ldexp(v, (side ? 13 : 17) * (k % 4));
      case INFINITE: return !side && r == 200 && k == 3 ? INFINITY : v;
      default: return v;
    }
  }
};

int main(int argc, char** argv) {
  const bool run = argc > 1 && std::strcmp(argv[1], "run") == 0;
  bool good = true;
  for (int ks : {1, 4}) {   // the parts of a split sum never add what lies at C
    Case c = {"", 300, 200, 2500, GEMM_TB, 1, NORMAL, LONG, false, 1, 0.5};
    GemmTask g = task(c, nullptr, nullptr, nullptr, nullptr, 0, 0);
    g.ksplit = ks;
    g.sK = g.sC;
    F64Plan p;
    plan_f64(&g, 1, p);
    for (const auto& l : p.t)
      for (const auto& t : l)
        if (t.beta != (ks == 1 ? 0.5 : 0.0)) { printf("%d splits: beta %g\n", ks, t.beta); good = false; }
  }
  for (const Case& c : CASES) {
    int nkr = 0, kv = c.k;
    std::vector<int> kr;
    if (c.runs) kr = run_table(c.k, nkr, kv);
    F64Plan p;
    good &= plan_holds(c, p, c.runs ? kr.data() : nullptr, nkr, kv);
    if (!run) continue;
    const size_t nA = (size_t)c.batch * c.m * c.k, nB = (size_t)c.n * c.k, nC = (size_t)c.batch * c.m * c.n;
    std::vector<double> X(nA), Y(nB), A(nA), B(nB), C0(nC), C(nC);
    Fill fill{std::mt19937_64(7), {}};
    for (int r = 0; r < c.batch * c.m; ++r)   // rows of X (batch entry, row), element k
      for (int k = 0; k < c.k; ++k) {
        const double v = X[(size_t)r * c.k + k] = fill(c.data, 0, r, k, c.k);
        const int b = r / c.m, i = r % c.m;
        A[(size_t)b * c.m * c.k + (c.flags & GEMM_TA ? (size_t)k * c.m + i : (size_t)i * c.k + k)] = v;
      }
    for (int r = 0; r < c.n; ++r)
      for (int k = 0; k < c.k; ++k) {
        const double v = Y[(size_t)r * c.k + k] = fill(c.data, 1, r, k, c.k);
        B[c.flags & GEMM_TB ? (size_t)r * c.k + k : (size_t)k * c.n + r] = v;
      }
    for (auto& v : C0) v = fill.g(fill.rng);
    double *dA, *dB, *dC;
    int *dkr = nullptr, *err;
    void* dt;
    bool ok = cudaMalloc(&dA, nA * 8) == cudaSuccess && cudaMalloc(&dB, nB * 8) == cudaSuccess &&
              cudaMalloc(&dC, nC * 8) == cudaSuccess && cudaMalloc(&err, 4) == cudaSuccess;
    if (ok && c.runs) ok = cudaMalloc(&dkr, kr.size() * 4) == cudaSuccess;
    if (!ok) return printf("%s: no memory\n", c.name), 1;
    cudaMemcpy(dA, A.data(), nA * 8, cudaMemcpyHostToDevice);
    cudaMemcpy(dB, B.data(), nB * 8, cudaMemcpyHostToDevice);
    cudaMemcpy(dC, C0.data(), nC * 8, cudaMemcpyHostToDevice);
    cudaMemset(err, 0, 4);
    if (c.runs) cudaMemcpy(dkr, kr.data(), kr.size() * 4, cudaMemcpyHostToDevice);
    plan_holds(c, p, dkr, nkr, kv, dA, dB, dC);
    if (cudaMalloc(&dt, f64_plan_bytes(p)) != cudaSuccess) return printf("%s: no memory\n", c.name), 1;
    upload_f64(p, dt, 0);
    int sms = 0, gave_up = 0;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, 0);
    // outputs in doubt: summed where they are found, by the second kernel, and both
    const size_t room = f64_scratch_bytes(p);
    const size_t rooms[3] = {0, room, room ? 256 + (room - 256) / 3 : 0};
    void* ds = nullptr;
    if (cudaMalloc(&ds, room + 256) != cudaSuccess) return printf("%s: no memory\n", c.name), 1;
    cudaMemset(ds, 0, 256);
    F64Scratch scratch{ds, 0, 0};
    for (size_t bytes : rooms) {
      scratch.bytes = bytes;
      cudaMemcpy(dC, C0.data(), nC * 8, cudaMemcpyHostToDevice);
      launch_f64(p, dt, 0, sms, err, 0, 2000000000ull, &scratch);
      cudaMemcpy(C.data(), dC, nC * 8, cudaMemcpyDeviceToHost);
      cudaMemcpy(&gave_up, err, 4, cudaMemcpyDeviceToHost);
      if (cudaDeviceSynchronize() != cudaSuccess || gave_up) return printf("%s: launch failed (%d)\n", c.name, gave_up), 1;
      // The sum with error-free products and sums (twice the working precision).
      // A chain of n multiply-adds is within n 2^-53 S of the sum, S = sum |x y|;
      // one more rounding of S for each of: the reference, alpha, beta C and the
      // sum with it, and the sums of 1024 terms added up; 2^-1074 per term where
      // products leave the range.
      double worst = 0;
      for (size_t e = 0; e < nC; ++e) {
        const double* x = &X[e / c.n * c.k];
        const double* y = &Y[e % c.n * (size_t)c.k];
        double s = 0, lo = 0, S = 0;
        int terms = 0;
        for (int k = 0; k < c.k; ++k) {
          if (c.runs && k % 48 >= 24) continue;
          const double q = x[k] * y[k], ql = std::fma(x[k], y[k], -q);
          const double t = s + q, bb = t - s;
          lo += (s - (t - bb)) + (q - bb) + ql;
          s = t;
          S += std::fabs(q);
          ++terms;
        }
        const double ref = c.alpha * (s + lo) + c.beta * C0[e];
        const double rounds = terms + 6 + terms / 1024;
        const double tol = rounds * (0x1p-53 * (std::fabs(c.alpha) * S + std::fabs(c.beta * C0[e])) + 0x1p-1074);
        if (c.data == INFINITE && e / c.n == 200) {   // the row with the infinity, and no other
          if (std::isfinite(C[e])) { printf("%s: output %zu is finite\n", c.name, e); ok = false; }
          continue;
        }
        const double d = std::fabs(C[e] - ref);
        if (!(d <= tol)) {
          if (ok) printf("%s: output %zu is %.17g, not %.17g: off by %.3g, bound %.3g\n", c.name, e, C[e], ref, d, tol);
          ok = false;
        }
        worst = std::max(worst, tol > 0 ? d / tol : 0.0);
      }
      printf("%s, %zu bytes of records: largest error %.3g of the bound\n", c.name, bytes, worst);
      good &= ok;
    }
    for (void* q : {(void*)dA, (void*)dB, (void*)dC, (void*)err, dt, ds, (void*)dkr}) cudaFree(q);
  }
  return good ? 0 : 1;
}
