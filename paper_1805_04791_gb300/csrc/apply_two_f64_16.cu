// Two-step passes of the apply, FP64, first radix up to 16 (see vie_two.cuh).
#include "vie_two.cuh"

namespace vie {
vie_status two_pass_f64_16(int pass, const TwoPlan& p, const TwoArgs& a, cudaStream_t st) {
  return two_pass<double, 16>(pass, p, a, st);
}
}  // namespace vie
