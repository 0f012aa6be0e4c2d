// <w, dR/dtheta> on hexahedra (the parameter part of the adjoint).
#include "enp_op_dispatch.cuh"
#include "enp_paramvjp.cuh"

cudaError_t enp::launch_param_vjp(const OpParams& prm, const double* u, const double* w, double* part,
                                  double* dtheta, int batch, cudaStream_t s) {
  if (prm.dim != 3) return cudaErrorInvalidConfiguration;
#define ENP_PV(PP)                                                                           \
  case PP:                                                                                   \
    if (prm.NF == 2) return launch_pvjp_pn<PP, 2>(prm, u, w, part, dtheta, batch, s);        \
    if (prm.NF == 3) return launch_pvjp_pn<PP, 3>(prm, u, w, part, dtheta, batch, s);        \
    return cudaErrorInvalidConfiguration;
  switch (prm.p) { ENP_PV(1) ENP_PV(2) ENP_PV(3) ENP_PV(4) }
#undef ENP_PV
  return cudaErrorInvalidConfiguration;
}
cudaError_t enp::upload_tables_param(int p, const Tables& t) { return upload_const_tables(p, t); }
