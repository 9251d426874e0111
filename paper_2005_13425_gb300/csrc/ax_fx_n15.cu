// The fixed-point ax_e kernels for n = 15.
#include "ax_fx_kernel.cuh"

namespace nekgb {
template nb_status launch_fx_n<15>(nb_ctx *, const double *, double *, int);
template void fx_tables_n<15>(nb_ctx *);
}  // namespace nekgb
