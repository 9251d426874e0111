// The fixed-point ax_e kernels for n = 13, 14.
#include "ax_fx_kernel.cuh"

namespace nekgb {
template nb_status launch_fx_n<13>(nb_ctx *, const double *, double *, int);
template nb_status launch_fx_n<14>(nb_ctx *, const double *, double *, int);
template void fx_tables_n<13>(nb_ctx *);
template void fx_tables_n<14>(nb_ctx *);
}  // namespace nekgb
