// General sweeps (dscf_coop.cuh) of replicas of unlike row layouts, FP64.
#include "dscf_coop.cuh"

namespace dscf {

template <>
const void* coop_mixed<double>() { return (const void*)k_prop_coop<double, 0>; }

}  // namespace dscf
