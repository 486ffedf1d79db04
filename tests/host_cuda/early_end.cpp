// A solve that ends early, at every call that can fail in turn: nothing that it enqueued
// may be unfinished when it returns, and the destruction of the problem waits for what
// it waits for before it gives the first buffer back.
#include <cstdio>
#include <map>
#include <set>
#include <vector>

#include <cuda_runtime_api.h>

#include "fake_cuda.h"
#include "vie.h"

static long one(int mode, long k, int* bad) {
  fake::State& s = fake::state();
  void* const create_stream = (void*)0x10;
  void* const solve_stream = (void*)0x20;
  const int n = 4, L = 3 * n * n * n;
  std::vector<double> eps(2 * 9 * n * n * n), b(2 * L), J(2 * L);
  vie_problem* P = nullptr;
  s.fail_at = -1;
  s.ones = false;
  cudaGetLastError();  // what the run before left
  if (vie_problem_create(VIE_HELMHOLTZ, n, -1, 1, 3.0, eps.data(), nullptr, create_stream, &P) != VIE_OK) return -1;
  s.ones = true;
  s.log.clear();
  s.work = 0;
  s.fail_at = k;
  vie_solve_opts o = {};
  o.tol = 1e-10;
  o.restart = 6;
  o.max_outer = 3;
  o.max_inner = 20;
  o.inner_tol = 1e-5;
  o.mode = mode;
  o.nrhs = 1;
  const vie_status st = vie_solve(P, b.data(), J.data(), &o, nullptr, solve_stream);
  const long work = s.work;
  // every stream's last enqueued work is followed by a wait for that stream
  std::set<uintptr_t> open;
  std::set<uintptr_t> recorded;
  for (const fake::Call& c : s.log) {
    if (c.op <= fake::RECORD) open.insert(c.stream);
    if (c.op == fake::RECORD) recorded.insert(c.event);
    if (c.op == fake::STREAM_SYNC) open.erase(c.stream);
  }
  // (a solve that ends by itself may leave its private stream, which the caller's stream waited for)
  if (st != VIE_OK && st != VIE_ENOCONV && !open.empty()) {
    printf("mode %d, call %ld failed: %zu streams not waited for\n", mode, k, open.size());
    ++*bad;
  }
  s.log.clear();
  s.fail_at = -1;
  vie_problem_destroy(P);
  size_t first_free = s.log.size(), last_wait = 0;
  for (size_t i = 0; i < s.log.size(); ++i) {
    if (s.log[i].op == fake::FREE && first_free == s.log.size()) first_free = i;
    if (s.log[i].op == fake::EVENT_SYNC) {
      recorded.erase(s.log[i].event);
      last_wait = i;
    }
  }
  if (last_wait > first_free) {
    printf("mode %d, call %ld failed: buffers given back before the steps' events are waited for\n", mode, k);
    ++*bad;
  }
  return work > k ? 1 : 0;
}

int main() {
  int bad = 0, runs = 0;
  const int modes[] = {VIE_SOLVE_MIXED, VIE_SOLVE_FP64, VIE_SOLVE_BICGSTAB};
  for (int mode : modes)
    for (long k = 0;; ++k, ++runs) {
      const long more = one(mode, k, &bad);
      if (more < 0) return 2;
      if (!more) break;
    }
  printf("%d runs, %d faults\n", runs, bad);
  return bad != 0;
}
