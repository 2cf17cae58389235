// An expired wait of any product reaches the caller: the report of a product that
// gave up is planted in the context, as the device would leave it, before a call
// or at one of the call's allocations, and the call must return
// MPSLCC_E_TIMEOUT; the same call then succeeds.  Exits 0 when every case holds.
#include <cmath>
#include <cstdio>
#include <functional>
#include <vector>

#include "engine.hpp"
#include "mpslcc.h"

using namespace mpslcc;

struct Plant {
  Ctx* c = nullptr;
  long count = 0, at = -1;
  int flag = 0;
};

static void* take(size_t n, void* user) {
  Plant* p = (Plant*)user;
  if (p->c && p->at == p->count++) p->c->out->flag[p->flag] = 99;
  void* q = nullptr;
  return cudaMalloc(&q, n) == cudaSuccess ? q : nullptr;
}
static void give(void* q, size_t, void* user) {
  Plant* p = (Plant*)user;
  if (p->c) cudaStreamSynchronize(p->c->s());
  cudaFree(q);
}

static int bad = 0;
static void expect(const char* what, int got, int want) {
  if (got == MPSLCC_E_NOCONV) got = MPSLCC_OK;   // the call completed
  if (got != want) {
    printf("%s: status %d, not %d\n", what, got, want);
    bad = 1;
  }
}

int main() {
  const int k = 6, ne = 6;
  Plant plant;
  mpslcc_opts o;
  mpslcc_default_opts(&o);
  o.alloc = take;
  o.free = give;
  o.alloc_user = &plant;
  o.tol = 1e-9;
  mpslcc_ctx* ctx = nullptr;
  if (mpslcc_create(&ctx, &o) != MPSLCC_OK) return printf("no context\n"), 1;
  Ctx* c = (Ctx*)ctx;   // its first member
  plant.c = c;
  // a Hubbard chain in its sites' basis
  std::vector<double> h(k * k, 0.0), V((size_t)k * k * k * k, 0.0);
  for (int i = 0; i + 1 < k; ++i) h[i * k + i + 1] = h[(i + 1) * k + i] = -1.0;
  for (int i = 0; i < k; ++i) { h[i * k + i] = 0.3 * i; V[((i * k + i) * (size_t)k + i) * k + i] = 2.0; }
  double e;
  if (mpslcc_build_mpo(ctx, h.data(), V.data(), k, ne, 0) != MPSLCC_OK ||
      mpslcc_set_spaces(ctx, 1, 4) != MPSLCC_OK || mpslcc_dmrg_reference(ctx, 16, 2, &e) != MPSLCC_OK ||
      mpslcc_lcc_sweep(ctx, 32, 1, 1, &e) == MPSLCC_E_ARG)
    return printf("set-up: %s\n", mpslcc_last_error(ctx)), 1;

  // products of a mixed-precision call on FP64 environments, either kind giving up
  long n = 0, m = 0;
  mpslcc_local_dim(ctx, 2, MPSLCC_OP_H0_11, &n, &m);
  std::vector<double> x(m, 1.0 / std::sqrt((double)m)), y(n), y0(n);
  for (int prec : {MPSLCC_FP64, MPSLCC_BF16X3, MPSLCC_BF16X6, MPSLCC_TF32}) {
    expect("apply", mpslcc_apply_heff(ctx, 2, MPSLCC_OP_H0_11, x.data(), y0.data(), m, n, prec), MPSLCC_OK);
    for (int flag : {0, 1}) {
      c->out->flag[flag] = 99;
      expect("apply after an expired wait", mpslcc_apply_heff(ctx, 2, MPSLCC_OP_H0_11, x.data(), y.data(), m, n, prec),
             MPSLCC_E_TIMEOUT);
      expect("apply again", mpslcc_apply_heff(ctx, 2, MPSLCC_OP_H0_11, x.data(), y.data(), m, n, prec), MPSLCC_OK);
      if (y != y0) { printf("apply again: another result\n"); bad = 1; }
    }
  }
  // calls that leave environments behind: the wait runs out at their last allocation
  const std::function<int()> calls[] = {
      [&] { return mpslcc_lcc_sweep_window(ctx, 32, 1, 0, 2, 1, &e); },
      [&] { return mpslcc_lcc_sweep_window(ctx, 32, 1, 1, 2, -1, &e); },
      [&] { return mpslcc_lcc_sweep(ctx, 32, 1, 1, &e); },
      [&] { return mpslcc_lcc_sweep_onesite(ctx, 1, 1, &e); },
      [&] { return mpslcc_dmrg_reference(ctx, 16, 1, &e); },
  };
  const char* names[] = {"window right", "window left", "sweep", "one-site sweep", "reference"};
  for (int i = 0; i < 5; ++i) {
    // run until the counts of two runs agree: the planted one makes the same allocations
    long before = -1, now = -2;
    for (int r = 0; r < 4 && before != now; ++r) {
      before = now;
      plant.count = 0;
      expect(names[i], calls[i](), MPSLCC_OK);
      now = plant.count;
    }
    for (long back = 1; back <= 2; ++back) {
      plant.count = 0;
      plant.at = now - back;
      const int st = calls[i]();
      const bool reached = plant.count > plant.at;
      plant.at = -1;
      expect(names[i], st, reached ? MPSLCC_E_TIMEOUT : MPSLCC_OK);
      if (!reached) printf("%s: made %ld allocations, not %ld\n", names[i], plant.count, now);
      expect("the call again", calls[i](), MPSLCC_OK);
    }
  }
  // a call that fails for another reason reports that one and leaves nothing behind
  c->out->flag[0] = 99;
  expect("wrong length", mpslcc_apply_heff(ctx, 2, MPSLCC_OP_H0_00, x.data(), y.data(), 1, 1, MPSLCC_FP64), MPSLCC_E_ARG);
  expect("energy of the reference", mpslcc_dmrg_reference(ctx, 16, 0, &e), MPSLCC_OK);
  plant.c = nullptr;
  mpslcc_destroy(ctx);
  return bad;
}
