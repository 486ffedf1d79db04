// What the library keeps between problems: bounded, given back when it is asked for, when an
// allocation fails and when the device is nearly full; nothing of a problem is left behind.
#include <cuda_runtime_api.h>

#include <cstdio>
#include <vector>

#include "fake_cuda.h"
#include "vie.h"

static int g_bad = 0;
#define CHECK(c)                                   \
  do {                                             \
    if (!(c)) {                                    \
      printf("line %d: %s\n", __LINE__, #c);       \
      ++g_bad;                                     \
    }                                              \
  } while (0)

static vie_status create(int n, vie_problem** P) {
  static const std::vector<double> eps(2 * 9 * 32 * 32 * 32);
  return vie_problem_create(VIE_HELMHOLTZ, n, -1, 1, 3.0, eps.data(), nullptr, nullptr, P);
}
static vie_status solve(vie_problem* P, int n) {
  std::vector<double> b(2 * 3 * n * n * n), J(b);
  vie_solve_opts o = {};
  o.tol = 1e-10;
  o.restart = 20;
  o.max_outer = 2;
  o.max_inner = 20;
  o.inner_tol = 1e-5;
  o.mode = VIE_SOLVE_MIXED;
  o.nrhs = 1;
  return vie_solve(P, b.data(), J.data(), &o, nullptr, nullptr);
}
// One request; the most bytes it held.
static size_t request(int n) {
  fake::State& s = fake::state();
  vie_problem* P = nullptr;
  s.high = s.live;
  const vie_status a = create(n, &P), b = a == VIE_OK ? solve(P, n) : a;
  CHECK(a == VIE_OK && (b == VIE_OK || b == VIE_ENOCONV));
  vie_problem_destroy(P);
  CHECK(s.live == 0);
  return s.high;
}

int main() {
  fake::State& s = fake::state();
  s.total = 1ull << 30;
  s.ones = true;
  // bounded by a thirty-second of the device
  CHECK(request(32) > s.total / 32);
  CHECK(s.threshold == s.total / 32 && s.kept > 0 && s.kept <= s.total / 32);
  // given back on request, pinned blocks included
  CHECK(s.host_blocks == 1);
  CHECK(vie_release_memory() == VIE_OK);
  CHECK(s.kept == 0 && s.host_blocks == 0);
  // an allocation that fails for what the pool keeps is tried again without it
  const size_t need = request(24);
  CHECK(s.kept > 0);
  const size_t total = s.total;
  s.total = need + s.kept / 2;
  s.trims = s.refused = 0;
  CHECK(request(24) == need);
  CHECK(s.refused == 1 && s.trims >= 1);
  // ... and one that fails for good returns VIE_ENOMEM and leaves nothing
  s.total = need / 2;
  cudaGetLastError();
  vie_problem* P = nullptr;
  vie_status st = create(24, &P);
  if (st == VIE_OK) st = solve(P, 24);
  CHECK(st == VIE_ENOMEM);
  vie_problem_destroy(P);
  CHECK(s.live == 0);
  // less than an eighth of the device free when a problem is destroyed: all goes back
  cudaGetLastError();
  s.total = total;
  vie_release_memory();
  CHECK(create(16, &P) == VIE_OK);
  s.foreign = s.total - s.live - s.total / 16;
  s.trims = 0;
  vie_problem_destroy(P);
  CHECK(s.trims == 1 && s.kept == 0);
  return g_bad != 0;
}
