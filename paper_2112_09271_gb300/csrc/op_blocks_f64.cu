// Assembly of the element-diagonal blocks, f64 arithmetic.
#include "enp_op_dispatch.cuh"
#include "enp_assemble.cuh"
ENP_ASSEMBLE_TYPE(double, c_paird)

template cudaError_t enp::launch_assemble<double>(const OpParams&, const io_t<double>*, io_t<double>*, cudaStream_t);
template cudaError_t enp::upload_tables_assemble<double>(int, const Tables&);
