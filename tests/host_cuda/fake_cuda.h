// A CUDA runtime that runs nothing: device memory is host memory, kernels and copies to
// the device do nothing, and every call that matters to ordering or memory is recorded.
// Host code linked against it (instead of the CUDA runtime) can be checked without a
// GPU, with any call made to fail.
#pragma once

#include <cstddef>
#include <cstdint>
#include <vector>

namespace fake {

enum Op { LAUNCH, COPY, MEMSET, RECORD, FREE, STREAM_SYNC, EVENT_SYNC, STREAM_WAIT };

struct Call {
  Op op;
  uintptr_t stream;  // of LAUNCH, COPY, MEMSET, RECORD, FREE, STREAM_SYNC, STREAM_WAIT
  uintptr_t event;   // of RECORD, EVENT_SYNC, STREAM_WAIT
};

struct State {
  std::vector<Call> log;
  long work = 0;         // launches, copies, memsets and event records so far
  long fail_at = -1;     // the work call (counted from `work`) that fails; -1: none
  bool ones = false;     // copies of reduction results to the host read as 1.0
  size_t live = 0, high = 0;    // device bytes allocated now, and at most
  size_t kept = 0;              // bytes given back that the pool still holds (never used again)
  size_t threshold = 0;         // of the pool: what it may hold when a stream is waited for
  size_t foreign = 0;           // bytes of other users of the device
  size_t total = 1ull << 38;    // bytes of the device
  long allocations = 0;         // calls so far, the ones that failed included
  long refuse_at = -1;          // the allocation that fails, tried twice in a row; -1: none
  int trims = 0, refused = 0;   // calls that gave kept bytes back, allocations that failed
  int host_blocks = 0;          // pinned blocks allocated now
};
State& state();

}  // namespace fake
