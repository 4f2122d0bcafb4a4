// Instances of the on-chip inner solve (res_kernels.cuh), in a translation
// unit of their own so that they compile beside the engine.
#include "engine.h"
#include "res_kernels.cuh"

namespace heat {

ResFn res_kernel(bool fp64, int elem) {
  if (fp64) return elem == E_P1 ? k_cg_res64<E_P1> : k_cg_res64<E_Q1>;
  return elem == E_P1 ? k_cg_res<E_P1> : k_cg_res<E_Q1>;
}

}  // namespace heat
