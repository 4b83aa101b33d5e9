// General contour sweeps (dscf_coop.cuh), FP32, and what the host needs to know of them.
#include "dscf_coop.cuh"

namespace dscf {

long long coop_units(const Rep& R) { return (long long)R.ny * R.nz * (R.nx <= 256 ? 1 : (R.nx + kCoopTile - 1) / kCoopTile); }

// CTAs of a launch: one per SM, fewer where that would leave a warp less than two row planes.
int coop_ctas(long long units, int nsm) {
    const long long w = 2LL * kCoopWarps;
    const long long n = (units + w - 1) / w;
    return (int)(n < 1 ? 1 : (n < nsm ? n : nsm));
}
int coop_warps_per_cta() { return kCoopWarps; }

CoopRep coop_rep(const Rep& R, int cost0) {
    CoopRep c = {};
    c.nx = R.nx; c.ny = R.ny; c.nz = R.nz; c.N = R.N; c.nA = R.nA;
    c.layout = coop_layout(R.nx);
    c.cost0 = cost0;
    c.units = (int)coop_units(R);
    c.V = R.V;
    c.E = R.E; c.G = R.G; c.Gp0 = R.Gp0; c.Gp1 = R.Gp1; c.q = R.q;
    c.qrow = R.qrow;
    c.pq = R.part + (size_t)P_Q * R.part_stride;
    c.qsum = R.scal + S_QSUM;
    c.rr = R.alpha / (1.0 - 2.0 * R.alpha);
    return c;
}

template int coop_prepare<float>(int);
template int launch_prop_coop<float>(const Launch&, const CoopPlan&, int, int, int);

}  // namespace dscf
