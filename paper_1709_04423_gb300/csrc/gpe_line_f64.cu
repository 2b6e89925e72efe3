// gpe_line_f64.cu -- instantiates the one-launch stepping of 1d grids for the double state.
#include "gpe_line.cuh"

namespace gpe {

bool takes_line_f64(const gp_handle* h) { return line_plan<double>(h->n[0] - 2).S > 0; }

int run_line_f64(gp_handle* h, bool imag, long nsteps) { return run_line_t<double>(h, imag, nsteps); }

}  // namespace gpe
