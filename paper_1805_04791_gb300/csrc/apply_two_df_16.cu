// Two-step passes of the apply, double-word, first radix up to 16 (see vie_two.cuh).
#include "vie_two.cuh"

namespace vie {
vie_status two_pass_df_16(int pass, const TwoPlan& p, const TwoArgs& a, cudaStream_t st) {
  if (pass == 3) return two_z_df_16(p, a, st);
  if (pass == 5) return two_last_pass<df, 16>(p, a, st);
  return two_line_pass<df, 16>(pass, p, a, st);
}
}  // namespace vie
