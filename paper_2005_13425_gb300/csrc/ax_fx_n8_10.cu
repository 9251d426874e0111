// The fixed-point ax_e kernels for n = 8, 9, 10.
#include "ax_fx_kernel.cuh"

namespace nekgb {
template nb_status launch_fx_n<8>(nb_ctx *, const double *, double *, int);
template nb_status launch_fx_n<9>(nb_ctx *, const double *, double *, int);
template nb_status launch_fx_n<10>(nb_ctx *, const double *, double *, int);
template void fx_tables_n<8>(nb_ctx *);
template void fx_tables_n<9>(nb_ctx *);
template void fx_tables_n<10>(nb_ctx *);
}  // namespace nekgb
