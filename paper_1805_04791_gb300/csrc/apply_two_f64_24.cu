// Two-step passes of the apply, FP64, first radix above 16 (see vie_two.cuh).
#include "vie_two.cuh"

namespace vie {
vie_status two_pass_f64_24(int pass, const TwoPlan& p, const TwoArgs& a, cudaStream_t st) {
  return two_pass<double, 24>(pass, p, a, st);
}
}  // namespace vie
