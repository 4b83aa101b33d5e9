// General contour sweeps (dscf_coop.cuh), FP64.
#include "dscf_coop.cuh"

namespace dscf {

template int coop_prepare<double>(int);
template int launch_prop_coop<double>(const Launch&, const CoopPlan&, int, int, int);

}  // namespace dscf
