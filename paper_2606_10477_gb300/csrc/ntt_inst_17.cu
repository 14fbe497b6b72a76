// Instantiations of the transform kernels for N = 2^17 (see ntt_impl.cuh).
#include "ntt_impl.cuh"

namespace hedap {

void ntt_launch_17(int v, const LimbSet& S, const Tables& T, cudaStream_t st, bool inverse, const NttAux& A,
                   const KskFuse* F) {
  launch_variant<9, 8>(v, S, T, st, inverse, A, F);
}

}  // namespace hedap
