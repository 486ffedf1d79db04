// vie_problem_bytes against the most device memory that a problem of the shape holds at
// a time: created, solved in mixed precision, its field evaluated.
#include <cstdio>
#include <vector>

#include "fake_cuda.h"
#include "vie.h"

int main() {
  fake::State& s = fake::state();
  int bad = 0;
  for (int kind : {VIE_LAPLACE, VIE_HELMHOLTZ, VIE_MAXWELL})
    for (int mu = 0; mu <= (kind == VIE_MAXWELL); ++mu)
      for (int n : {16, 24, 31, 48, 62})
        for (int nrhs : {1, 3})
          for (int restart : {5, 30}) {
            const size_t c = mu ? 6 : 3, N = (size_t)n * n * n;
            std::vector<double> eps(2 * 9 * N), b(2 * c * N * nrhs), J(b), f(2 * 6 * N * nrhs);
            vie_problem* P = nullptr;
            s.high = s.live;
            s.ones = false;
            vie_status st = vie_problem_create(kind, n, -1, 1, kind == VIE_LAPLACE ? 0.0 : 3.0, eps.data(),
                                               mu ? eps.data() : nullptr, nullptr, &P);
            const size_t created = s.high;
            s.ones = true;
            vie_solve_opts o = {};
            o.tol = 1e-10;
            o.restart = restart;
            o.max_outer = 2;
            o.max_inner = 2 * restart;
            o.inner_tol = 1e-5;
            o.mode = VIE_SOLVE_MIXED;
            o.nrhs = nrhs;
            if (st == VIE_OK) st = vie_solve(P, b.data(), J.data(), &o, nullptr, nullptr);
            const size_t solved = s.high;
            if (st == VIE_OK || st == VIE_ENOCONV) st = vie_eval_scattered(P, J.data(), f.data(), nrhs, nullptr);
            const size_t most = s.high, said = vie_problem_bytes(kind, n, nrhs, restart, mu);
            vie_problem_destroy(P);
            const bool ok = st == VIE_OK && said >= most && said <= most + most / 20 + (256 << 10);
            if (!ok) ++bad;
            printf("%s kind %d mu %d n %d nrhs %d restart %d: %zu bytes said, %zu held (created %zu, solved %zu)\n",
                   ok ? "ok " : "BAD", kind, mu, n, nrhs, restart, said, most, created, solved);
          }
  return bad != 0;
}
