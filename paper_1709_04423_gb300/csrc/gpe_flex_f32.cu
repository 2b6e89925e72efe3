// gpe_flex_f32.cu -- instantiates the sweeps on tiles of few lines for the float state.
#include "gpe_flex.cuh"

namespace gpe {

template <>
void run_flex<float>(const Sweep2Args<float>& a, const FlexPlan& p, bool imag, bool last, bool close, bool var,
                  cudaStream_t s, bool pdl) {
  run_flex_t<float>(a, p, imag, last, close, var, s, pdl);
}

}  // namespace gpe
