// Forward density map phi[U] without any device allocation by the caller or the library.
//
// Some callers cannot call cudaMalloc (or any allocator) at all: code running inside a host
// framework that owns every device allocation and hands out only its own buffers, plug-ins
// invoked from a callback where allocation is forbidden, or processes that must not grow their
// device footprint after start-up.  They cannot provide the workspace the context-based API
// needs.  This entry point takes only the input potentials and the output densities; the
// propagator stack, Boltzmann factors, quadratures, partial sums and replica table live in one
// file-scope device array of fixed size, which every GPU that loads this code keeps for the life
// of the process.
#include <cuda_runtime.h>

#include <cstring>
#include <mutex>

#include "../../include/dscf.h"
#include "dscf_internal.cuh"

using namespace dscf;

namespace dscf {
void set_thread_error(const char* msg);
}

namespace {

static __device__ __align__(256) unsigned char g_scratch[DSCF_STATIC_SCRATCH_BYTES];

constexpr int kMaxDevices = 64;
std::mutex g_mu;
unsigned char* g_scratch_dev[kMaxDevices] = {};   // device address of g_scratch, per device

size_t up256(size_t x) { return (x + 255) & ~(size_t)255; }

// Writes the replica descriptors into the scratch; passed by value so no host-to-device copy (and no
// staging buffer) is needed.
__global__ void k_put_rep(Rep* dst, Rep r, CoopRep* dstc, CoopRep c) {
    *dst = r;
    *dstc = c;
}

}  // namespace

namespace {
int densities_static_on(const dscf_params* p, int32_t precision, const void* U_in, void* phi_out, void* stream);
}

// Runs on the device that holds U_in and leaves the calling thread's current device as it found it.
extern "C" int dscf_densities_static(const dscf_params* p, int32_t precision, const void* U_in, void* phi_out,
                                     void* stream) {
    int prev = -1;
    if (cudaGetDevice(&prev) != cudaSuccess) {
        cudaGetLastError();
        set_thread_error("dscf_densities_static: cudaGetDevice failed");
        return DSCF_ERR_CUDA;
    }
    const int rc = densities_static_on(p, precision, U_in, phi_out, stream);
    if (cudaSetDevice(prev) != cudaSuccess && rc == DSCF_OK) {
        set_thread_error("dscf_densities_static: restoring the caller's device failed");
        return DSCF_ERR_CUDA;
    }
    return rc;
}

namespace {
int densities_static_on(const dscf_params* p, int32_t precision, const void* U_in, void* phi_out, void* stream) {
    if (!p || !U_in || !phi_out) {
        set_thread_error("dscf_densities_static: NULL argument");
        return DSCF_ERR_ARG;
    }
    if (precision != DSCF_FP64 && precision != DSCF_FP32) {
        set_thread_error("dscf_densities_static: bad precision");
        return DSCF_ERR_ARG;
    }
    if (dscf_workspace_bytes(p, 1, precision) == 0) {
        set_thread_error("dscf_densities_static: invalid parameters");
        return DSCF_ERR_ARG;
    }
    // the device that holds the input selects the copy of the scratch array
    cudaPointerAttributes pa;
    if (cudaPointerGetAttributes(&pa, U_in) != cudaSuccess || pa.type != cudaMemoryTypeDevice) {
        cudaGetLastError();
        set_thread_error("dscf_densities_static: U_in is not device memory");
        return DSCF_ERR_ARG;
    }
    const int dev = pa.device;
    if (dev < 0 || dev >= kMaxDevices) {
        set_thread_error("dscf_densities_static: device index out of range");
        return DSCF_ERR_ARG;
    }
    if (cudaSetDevice(dev) != cudaSuccess) {
        set_thread_error("dscf_densities_static: cudaSetDevice failed");
        return DSCF_ERR_CUDA;
    }

    // Tiling of one replica, as the context-based path does it.
    const size_t es = precision == DSCF_FP64 ? sizeof(double) : sizeof(float);
    Rep R;
    std::memset(&R, 0, sizeof R);
    R.nx = p->nx; R.ny = p->ny; R.nz = p->nz; R.ns = p->ns; R.N = p->N; R.nA = p->nA;
    R.V = (long long)p->nx * p->ny * p->nz;
    tile_replica(R);
    R.phi_p = p->phi_p;
    R.alpha = p->a * p->a / 6.0;
    set_pars(R);
    int nsm = 0;
    if (cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
        set_thread_error("dscf_densities_static: device query failed");
        return DSCF_ERR_CUDA;
    }
    if (nsm > kCoopMaxCtas) nsm = kCoopMaxCtas;
    CoopPlan plan;
    plan.nrep = 1;
    plan.kk = coop_layout(R.nx, R.V, precision == DSCF_FP64);
    coop_cut(plan, R, coop_units(R, precision == DSCF_FP64), precision == DSCF_FP64, nsm);
    // Scratch layout: replica table, maps, Boltzmann factors, propagators, quadratures,
    // partial sums, scalars.
    const size_t V = (size_t)R.V;
    size_t off, o_rep, o_coop, o_b2r, o_E, o_G, o_Gp0, o_Gp1, o_q, o_part, o_scal;
    for (;;) {
        R.nq = plan.ncta * coop_warps(plan.kk, precision == DSCF_FP64);
        R.part_stride = R.nq > R.nblk ? R.nq : R.nblk;
        off = 0;
        auto take = [&](size_t bytes) { const size_t o = off; off = up256(off + bytes); return o; };
        o_rep = take(sizeof(Rep));
        o_coop = take(sizeof(CoopRep));
        o_b2r = take(sizeof(int) * R.nblk);
        o_E = take((size_t)R.ns * V * es);
        o_G = take((size_t)R.N * V * es);
        o_Gp0 = take(V * es);
        o_Gp1 = take(V * es);
        o_q = take(2 * V * es);
        o_part = take(sizeof(double) * 2 * (size_t)R.part_stride);   // P_Q, P_ES
        o_scal = take(sizeof(double) * kScalStride);
        if (off <= (size_t)DSCF_STATIC_SCRATCH_BYTES || plan.ncta == 1) break;
        plan.ncta = (plan.ncta + 1) / 2;   // near the limit: fewer warps' partial sums, an even cut
        plan.runs = plan.per = 0;
    }
    if (off > (size_t)DSCF_STATIC_SCRATCH_BYTES) {
        set_thread_error("dscf_densities_static: the problem needs more scratch than DSCF_STATIC_SCRATCH_BYTES");
        return DSCF_ERR_OOM;
    }

    // Set-up, once per device: the host-side name g_scratch is only a stand-in, the kernels need
    // the device address of this device's copy.
    unsigned char* base = nullptr;
    {
        std::lock_guard<std::mutex> lock(g_mu);
        if (!g_scratch_dev[dev]) {
            void* ptr = nullptr;
            cudaError_t e = cudaGetSymbolAddress(&ptr, g_scratch);
            if (e != cudaSuccess || !ptr) {
                set_thread_error("dscf_densities_static: cudaGetSymbolAddress failed");
                return DSCF_ERR_CUDA;
            }
            g_scratch_dev[dev] = (unsigned char*)ptr;
        }
        base = g_scratch_dev[dev];
    }
    R.E = base + o_E;
    R.G = base + o_G;
    R.Gp0 = base + o_Gp0;
    R.Gp1 = base + o_Gp1;
    R.q = base + o_q;
    R.part = (double*)(base + o_part);
    R.scal = (double*)(base + o_scal);
    R.blk0 = 0;
    R.ext_off = 0;
    R.vbase = 0;

    if ((precision == DSCF_FP64 ? coop_prepare<double>(plan.kk) : coop_prepare<float>(plan.kk)) != 0) {
        set_thread_error("dscf_densities_static: the contour kernels do not load");
        return DSCF_ERR_CUDA;
    }

    cudaStream_t s = (cudaStream_t)stream;
    Launch L;
    L.reps = (const Rep*)(base + o_rep);
    L.blk2rep = (const int*)(base + o_b2r);
    L.status = nullptr;
    L.counter = nullptr;
    L.nblk_total = R.nblk;
    L.nlb_total = R.lb_nblk;
    L.nrep = 1;
    L.stream = s;
    plan.reps = (const CoopRep*)(base + o_coop);
    plan.cnt = plan.abort = nullptr;   // one level per launch: no barrier inside a launch
    // the only state that must start at zero: the block map (one replica, index 0)
    cudaError_t e = cudaMemsetAsync(base + o_b2r, 0, sizeof(int) * R.nblk, s);
    if (e != cudaSuccess) {
        set_thread_error("dscf_densities_static: cudaMemsetAsync failed");
        return DSCF_ERR_CUDA;
    }
    k_put_rep<<<1, 1, 0, s>>>((Rep*)(base + o_rep), R, (CoopRep*)(base + o_coop), coop_rep(R, precision == DSCF_FP64, 1, 0));
    if (precision == DSCF_FP64) {
        launch_exp<double>(L, 3, 0, U_in);
        for (int j = 0; j < R.N; ++j) launch_prop_coop<double>(L, plan, j, j + 1, 1);
        launch_dens_out<double>(L, phi_out);
    } else {
        launch_exp<float>(L, 3, 0, U_in);
        for (int j = 0; j < R.N; ++j) launch_prop_coop<float>(L, plan, j, j + 1, 1);
        launch_dens_out<float>(L, phi_out);
    }
    e = cudaGetLastError();
    if (e != cudaSuccess) {
        set_thread_error(cudaGetErrorString(e));
        return DSCF_ERR_CUDA;
    }
    return DSCF_OK;
}
}  // namespace
