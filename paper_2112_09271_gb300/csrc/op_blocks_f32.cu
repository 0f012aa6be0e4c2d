// Assembly of the element-diagonal blocks, f32 arithmetic.
#include "enp_op_dispatch.cuh"
#include "enp_assemble.cuh"
ENP_ASSEMBLE_TYPE(float, c_pairf)

template cudaError_t enp::launch_assemble<float>(const OpParams&, const io_t<float>*, io_t<float>*, cudaStream_t);
template cudaError_t enp::upload_tables_assemble<float>(int, const Tables&);
