// Inverses of the element blocks of hexahedra by elimination of the species.
#include "enp_blockinv.cuh"
#include "enp_internal.h"

bool enp::elimination_available(int dim, int p) { return dim == 3 && p >= 2 && p <= 4; }

cudaError_t enp::launch_elimination(float* blocks, void* out, int storage, int p, int nf,
                                    long long nblk, int* singular, cudaStream_t s) {
  if ((nf != 2 && nf != 3) || (storage != 1 && storage != 2)) return cudaErrorInvalidConfiguration;
  switch (p) {
    case 2: return nf == 2 ? launch_elim_n<27, 1, 1, 2>(blocks, out, storage, nblk, singular, s)
                           : launch_elim_n<27, 1, 1, 3>(blocks, out, storage, nblk, singular, s);
    case 3: return nf == 2 ? launch_elim_n<64, 1, 2, 2>(blocks, out, storage, nblk, singular, s)
                           : launch_elim_n<64, 1, 2, 3>(blocks, out, storage, nblk, singular, s);
    case 4: return nf == 2 ? launch_elim_n<125, 4, 1, 2>(blocks, out, storage, nblk, singular, s)
                           : launch_elim_n<125, 4, 1, 3>(blocks, out, storage, nblk, singular, s);
  }
  return cudaErrorInvalidConfiguration;
}
