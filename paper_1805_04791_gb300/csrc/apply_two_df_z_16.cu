// Two-step z pass of the apply, double-word, first radix up to 16 (see vie_two.cuh).
#include "vie_two.cuh"

namespace vie {
vie_status two_z_df_16(const TwoPlan& p, const TwoArgs& a, cudaStream_t st) { return two_z_pass<df, 16>(p, a, st); }
}  // namespace vie
