// gpe_line_f64.cu -- instantiates the one-launch stepping of 1d grids for the double state.
#include "gpe_line.cuh"

namespace gpe {

int run_line_f64(gp_handle* h, bool imag, long nsteps) { return run_line_t<double>(h, imag, nsteps); }

}  // namespace gpe
