// gpe_flex_f64.cu -- instantiates the sweeps on tiles of few lines for the double state.
#include "gpe_flex.cuh"

namespace gpe {

template <>
void run_flex<double>(const Sweep2Args<double>& a, const FlexPlan& p, bool imag, bool last, bool close, bool var,
                  cudaStream_t s, bool pdl) {
  run_flex_t<double>(a, p, imag, last, close, var, s, pdl);
}

}  // namespace gpe
