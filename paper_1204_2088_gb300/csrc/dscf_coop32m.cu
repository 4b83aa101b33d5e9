// General sweeps (dscf_coop.cuh) of replicas of unlike row layouts, FP32.
#include "dscf_coop.cuh"

namespace dscf {

template <>
const void* coop_mixed<float>() { return (const void*)k_prop_coop<float, 0>; }

}  // namespace dscf
