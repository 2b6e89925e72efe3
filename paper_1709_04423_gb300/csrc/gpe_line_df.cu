// gpe_line_df.cu -- instantiates the one-launch stepping of 1d grids for the df64 state.
#include "gpe_line.cuh"

namespace gpe {

bool takes_line_df(const gp_handle* h) { return line_plan<df64>(h->n[0] - 2).S > 0; }

int run_line_df(gp_handle* h, bool imag, long nsteps) { return run_line_t<df64>(h, imag, nsteps); }

}  // namespace gpe
