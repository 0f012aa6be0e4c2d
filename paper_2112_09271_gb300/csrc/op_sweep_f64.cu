// The downwind sweep on FP64 vectors.
#include "enp_op_dispatch.cuh"
#include "enp_sweep.cuh"

template cudaError_t enp::launch_sweep<double>(const OpParams&, const void*, int, const double*, double*,
                                         const double*, int, cudaStream_t, int, int, int, bool);
template <> cudaError_t enp::upload_tables_sweep<double>(int p, const Tables& t) {
  return upload_const_tables(p, t);
}
