// The fixed-point ax_e kernels for n = 11, 12.
#include "ax_fx_kernel.cuh"

namespace nekgb {
template nb_status launch_fx_n<11>(nb_ctx *, const double *, double *, int);
template nb_status launch_fx_n<12>(nb_ctx *, const double *, double *, int);
template void fx_tables_n<11>(nb_ctx *);
template void fx_tables_n<12>(nb_ctx *);
}  // namespace nekgb
