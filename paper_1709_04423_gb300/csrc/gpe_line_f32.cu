// gpe_line_f32.cu -- instantiates the one-launch stepping of 1d grids for the float state.
#include "gpe_line.cuh"

namespace gpe {

bool takes_line_f32(const gp_handle* h) { return line_plan<float>(h->n[0] - 2).S > 0; }

int run_line_f32(gp_handle* h, bool imag, long nsteps) { return run_line_t<float>(h, imag, nsteps); }

}  // namespace gpe
