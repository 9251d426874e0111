// The fixed-point ax_e kernels for n = 2, 3, 4, 5, 6, 7.
#include "ax_fx_kernel.cuh"

namespace nekgb {
template nb_status launch_fx_n<2>(nb_ctx *, const double *, double *, int);
template nb_status launch_fx_n<3>(nb_ctx *, const double *, double *, int);
template nb_status launch_fx_n<4>(nb_ctx *, const double *, double *, int);
template nb_status launch_fx_n<5>(nb_ctx *, const double *, double *, int);
template nb_status launch_fx_n<6>(nb_ctx *, const double *, double *, int);
template nb_status launch_fx_n<7>(nb_ctx *, const double *, double *, int);
template void fx_tables_n<2>(nb_ctx *);
template void fx_tables_n<3>(nb_ctx *);
template void fx_tables_n<4>(nb_ctx *);
template void fx_tables_n<5>(nb_ctx *);
template void fx_tables_n<6>(nb_ctx *);
template void fx_tables_n<7>(nb_ctx *);
}  // namespace nekgb
