// The downwind sweep on FP32 vectors.
#include "enp_op_dispatch.cuh"
#include "enp_sweep.cuh"

template cudaError_t enp::launch_sweep<float>(const OpParams&, const void*, int, const float*, float*,
                                         const float*, int, cudaStream_t, int, int, int, bool);
template <> cudaError_t enp::upload_tables_sweep<float>(int p, const Tables& t) {
  return upload_const_tables(p, t);
}
