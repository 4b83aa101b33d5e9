// General contour sweeps (dscf_coop.cuh), FP32, and what the host needs to know of them.
#include "dscf_coop.cuh"

#include <algorithm>

namespace dscf {

static int layout_of(const Rep& R, bool fp64) { return coop_layout(R.nx, R.V, fp64); }
static long long rows_of(const Rep& R, bool fp64) {
    const int g = coop_group(R.nx, R.V, fp64);
    return (long long)coop_tiles(R.nx) * ((R.ny + g - 1) / g);
}
long long coop_units(const Rep& R, bool fp64) { return rows_of(R, fp64) * R.nz; }

// Strips of 8 rows in fields of 2^23 sites and more, so that a CTA's warps share rows in the L1 at about the same
// time (256^3, N = 64: 7.93 -> 7.56 ms; levels of that size, FP32 or FP64, pass through the L2); up to 128^3
// sharing gains nothing (924 -> 984 us).
static int strip_rows(const Rep& R) { return R.V >= (1LL << 23) && R.ny % 8 == 0 && coop_warps(layout_of(R, false), false) == 8 ? 8 : 1; }

// Cut of a launch's work.  One replica whose rows can be cut into equal runs gives every warp one run
// (runs > 0): a warp of an even cut of all row planes mostly ends one row and begins another, which costs two
// more planes of the y and x passes and, in FP32, the loads' latency once more, and the slowest warp makes
// the level's time.  Density evaluations with the even cut and with runs: 100 x 90 x 75, N = 48, FP32 364 and
// 281 us; 64^3, N = 64, FP32 331 and 241; 32^3, N = 32, FP64 265 and 132.  The runs are spread over all SMs.
// Where whole runs would leave too many warps idle (estimated below in planes), and in batches, the cut is
// even, at least two row planes a warp.
void coop_cut(CoopPlan& c, const Rep& R, long long work, bool fp64, int nsm) {
    const int nw = coop_warps(c.kk, fp64), P = nsm * nw;
    c.runs = c.per = 0;
    if (c.nrep == 1) {
        const long long rows = rows_of(R, fp64);
        if (rows <= P) {
            int r = std::min((int)(P / rows), R.nz);
            const int n = (R.nz + r - 1) / r;
            r = (R.nz + n - 1) / n;
            const double even = (double)((work + P - 1) / P) + (fp64 ? 2.0 + 2.0 * rows / P : 8.0);
            if (n + (fp64 ? 2 : 4) <= even) {
                c.runs = r;
                c.per = (int)((rows * r + nsm - 1) / nsm);
                c.ncta = (int)((rows * r + c.per - 1) / c.per);
                return;
            }
        }
    }
    const long long w = 2LL * nw, n = (work + w - 1) / w;
    c.ncta = (int)(n < 1 ? 1 : (n < nsm ? n : nsm));
}

// a row plane's time: FP32 mostly the latency of its loads, FP64 mostly its operations
int coop_cost(const Rep& R, bool fp64) { return fp64 ? 1 + 2 * (layout_of(R, true) & 15) : 4 + (layout_of(R, false) & 15); }

CoopRep coop_rep(const Rep& R, bool fp64, int cost, int cost0) {
    CoopRep c = {};
    c.nx = R.nx; c.ny = R.ny; c.nz = R.nz; c.N = R.N; c.nA = R.nA;
    c.layout = (short)layout_of(R, fp64);
    c.cost0 = cost0;
    c.units = (int)coop_units(R, fp64);
    c.tile = coop_narrow(R.nx, R.V, fp64) ? coop_group(R.nx, R.V, fp64) : coop_tile(R.nx);
    c.strip = (short)strip_rows(R);
    c.wgt = cost * c.strip;
    c.V = R.V;
    c.E = R.E; c.G = R.G; c.Gp0 = R.Gp0; c.Gp1 = R.Gp1; c.q = R.q;
    c.qrow = R.qrow;
    c.pq = R.part + (size_t)P_Q * R.part_stride;
    c.qsum = R.scal + S_QSUM;
    c.rr = fp64 ? R.pd.rr : (double)R.pf.rr;
    return c;
}

template int coop_prepare<float>(int);
template int launch_prop_coop<float>(const Launch&, const CoopPlan&, int, int, int);

}  // namespace dscf
