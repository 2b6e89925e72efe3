// gpe_flex_df.cu -- instantiates the sweeps on tiles of few lines for the df64 state.
#include "gpe_flex.cuh"

namespace gpe {

template <>
void run_flex<df64>(const Sweep2Args<df64>& a, const FlexPlan& p, bool imag, bool last, bool close, bool var,
                  cudaStream_t s, bool pdl) {
  run_flex_t<df64>(a, p, imag, last, close, var, s, pdl);
}

}  // namespace gpe
