// The solvers' fused vector passes (kernels.cu) against the separate ones, bit
// for bit, and the dots against their stated order on the host.  Exits 0 when
// every case holds.
#include <cmath>
#include <cstdio>
#include <cstring>
#include <random>
#include <vector>

#include "kernels.hpp"

using namespace mpslcc;

static double tree(const double* v, int n) {   // shuffle-down tree over 32 lanes, zeros past n
  double a[32] = {};
  for (int i = 0; i < n; ++i) a[i] = v[i];
  for (int o = 16; o > 0; o >>= 1)
    for (int i = 0; i + o < 32; ++i) a[i] += a[i + o];
  return a[0];
}
static double block(const double* v) {
  double w[8];
  for (int i = 0; i < 8; ++i) w[i] = tree(v + 32 * i, 32);
  return tree(w, 8);
}
// the dot as `blocks` blocks of 256 threads take it
static double host_dot(const std::vector<double>& x, const std::vector<double>& y, int blocks) {
  std::vector<double> th(256 * (size_t)blocks, 0.0), part(std::max(256, blocks), 0.0), last(256, 0.0);
  for (size_t i = 0; i < x.size(); ++i) th[i % th.size()] = std::fma(x[i], y[i], th[i % th.size()]);
  for (int b = 0; b < blocks; ++b) part[b] = block(&th[256 * (size_t)b]);
  for (int i = 0; i < blocks; ++i) last[i % 256] += part[i];
  return block(last.data());
}

int main() {
  std::mt19937_64 rng(3);
  std::normal_distribution<double> g;
  double *part, *out;
  unsigned int* tk;
  const int M = 5;
  cudaMalloc(&part, 4096 * 8);
  cudaMalloc(&out, 64 * 8);
  cudaMalloc(&tk, MD_TICKETS * 4);
  cudaMemset(tk, 0, MD_TICKETS * 4);
  const Reduction R{part, tk, out};
  for (long n : {1L, 31L, 255L, 256L, 257L, 16384L, 16385L, 131071L, 131072L, 131073L, 300001L}) {
    auto vec = [&](long m) {
      std::vector<double> h(m);
      for (auto& v : h) v = g(rng);
      return h;
    };
    auto dev = [&](const std::vector<double>& h) {
      double* d = nullptr;
      cudaMalloc(&d, h.size() * 8);
      cudaMemcpy(d, h.data(), h.size() * 8, cudaMemcpyHostToDevice);
      return d;
    };
    auto host = [&](const double* d, long m) {
      std::vector<double> h(m);
      cudaMemcpy(h.data(), d, m * 8, cudaMemcpyDeviceToHost);
      return h;
    };
    auto same = [&](const double* a, const double* b, long m) {
      return std::memcmp(host(a, m).data(), host(b, m).data(), m * 8) == 0;
    };
    auto bad = [&](const char* w) { return std::printf("FAIL %s n=%ld\n", w, n), 1; };
    const auto hx = vec(n), hy = vec(n), hp = vec(n), hd = vec(n), hV = vec(M * n), hA = vec(M * n);
    double *p = dev(hp), *d = dev(hd), *V = dev(hV), *A = dev(hA);
    double *x1 = dev(hx), *x2 = dev(hx), *y1 = dev(hy), *y2 = dev(hy), *z1 = dev(hx), *z2 = dev(hx);
    // two dots
    launch_dot_fused(x1, y1, p, p, n, out, part, tk, 0);
    auto r = host(out, 2);
    if (r[0] != host_dot(hx, hy, 512) || r[1] != host_dot(hp, hp, 512)) return bad("dot");
    // y -= shift p; p.y
    launch_shift_dot(n, 0.37, p, y1, p, R, 0);
    launch_axpy(n, -0.37, p, y2, 0);
    if (!same(y1, y2, n)) return bad("shift");
    if (host(out, 1)[0] != host_dot(hp, host(y1, n), 512)) return bad("shift dot");
    // CG update
    launch_cg_update(n, 0.61, p, A, x1, y1, d, 0.2, 1e-2, z1, R, 0);
    r = host(out, 2);
    launch_axpy(n, 0.61, p, x2, 0);
    launch_axpy(n, -0.61, A, y2, 0);
    launch_precond(n, y2, d, 0.2, 1e-2, z2, 1, 0);
    if (!same(x1, x2, n) || !same(y1, y2, n) || !same(z1, z2, n)) return bad("cg");
    if (r[0] != host_dot(host(y2, n), host(z2, n), 512) || r[1] != host_dot(host(y2, n), host(y2, n), 512))
      return bad("cg dots");
    // Ritz vector and residual
    const double c[M] = {0.3, -0.8, 0.1, 0.45, -0.2};
    launch_ritz(n, M, V, A, n, c, -1.3, x1, y1, R, 0);
    r = host(out, 1);
    launch_lincomb_args(n, M, V, n, c, x2, 0);
    launch_lincomb_args(n, M, A, n, c, y2, 0);
    launch_axpy(n, 1.3, x2, y2, 0);
    if (!same(x1, x2, n) || !same(y1, y2, n)) return bad("ritz");
    if (r[0] != host_dot(host(y2, n), host(y2, n), 512)) return bad("ritz dot");
    // overlaps and the orthogonalisation with them
    launch_multidot(n, M, V, n, z1, out, part, tk, 0);
    r = host(out, M);
    for (int j = 0; j < M; ++j)
      if (r[j] != host_dot(std::vector<double>(hV.begin() + j * n, hV.begin() + (j + 1) * n), host(z1, n), 64))
        return bad("overlaps");
    launch_gs(n, M, V, n, out, z1, 0);
    for (auto& v : r) v = -v;
    launch_lincomb_args(n, M, V, n, r.data(), x2, 0);
    launch_axpy(n, 1.0, x2, z2, 0);
    if (!same(z1, z2, n)) return bad("orthogonalise");
    for (double* q : {p, d, V, A, x1, x2, y1, y2, z1, z2}) cudaFree(q);
  }
  if (cudaDeviceSynchronize() != cudaSuccess) return std::printf("FAIL device\n"), 1;
  std::printf("ok\n");
  return 0;
}
