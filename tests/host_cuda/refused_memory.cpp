// After an allocation that failed, at every allocation in turn: the call says so, and the
// same call and all later ones work once there is memory.
#include <cstdio>
#include <vector>

#include "fake_cuda.h"
#include "vie.h"

static int g_bad = 0;

// Applies in each precision and the field; with one allocation refused, the call that
// meets it is made again.  Returns the bytes held at the end, 0 if nothing was refused.
static size_t run(int kind, bool with_mu, long refuse) {
  fake::State& s = fake::state();
  const int n = 8, N = n * n * n, c = with_mu ? 6 : 3;
  std::vector<double> eps(2 * 9 * N), x(2 * c * N), y(x), f(2 * 6 * N);
  vie_problem* P = nullptr;
  if (vie_problem_create(kind, n, -1, 1, 3.0, eps.data(), with_mu ? eps.data() : nullptr, nullptr, &P) != VIE_OK) {
    printf("create failed\n");
    ++g_bad;
    return 0;
  }
  s.allocations = 0;
  s.refuse_at = refuse;
  bool refused = false;
  for (int call = 0; call < 4; ++call)
    for (int again = 0; again < 2; ++again) {
      const int prec[] = {VIE_FP64, VIE_DF64, VIE_FP32};
      const vie_status st = call < 3 ? vie_apply(P, x.data(), y.data(), prec[call], 1, nullptr)
                                     : vie_eval_scattered(P, x.data(), f.data(), 1, nullptr);
      if (st == VIE_OK) break;
      if (st != VIE_ENOMEM || refused) {
        printf("kind %d mu %d allocation %ld refused: call %d returned %d\n", kind, with_mu, refuse, call, (int)st);
        ++g_bad;
        break;
      }
      refused = true;
    }
  s.refuse_at = -1;
  const size_t held = s.live;
  vie_problem_destroy(P);
  if (s.live) {
    printf("kind %d mu %d allocation %ld refused: %zu bytes left\n", kind, with_mu, refuse, s.live);
    ++g_bad;
    s.live = 0;
  }
  return refused || refuse < 0 ? held : 0;
}

int main() {
  int runs = 0;
  for (int kind : {VIE_HELMHOLTZ, VIE_MAXWELL})
    for (int mu = 0; mu <= (kind == VIE_MAXWELL); ++mu) {
      const size_t whole = run(kind, mu, -1);
      for (long k = 0;; ++k, ++runs) {
        const size_t held = run(kind, mu, k);
        if (!held) break;
        if (held != whole) {
          printf("kind %d mu %d allocation %ld refused: %zu bytes held in the end, %zu without\n", kind, mu, k, held, whole);
          ++g_bad;
        }
      }
    }
  printf("%d runs, %d faults\n", runs, g_bad);
  return g_bad != 0 || runs < 10;
}
