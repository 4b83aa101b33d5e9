// Internal declarations of the CUDA library: replica descriptors, partial-sum slots and the
// deterministic block reductions every kernel uses.  Not part of the public ABI.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <cmath>

namespace dscf {

constexpr int kFlatThreads = 256;     // threads of every site-parallel ("flat") kernel
constexpr int kMaxFlatBlocks = 608;   // flat blocks per replica (= partial sums per replica): 4 per SM, one wave
constexpr int kMaxNcg = 32;           // Fletcher-Reeves iterations per step, upper bound
constexpr int kScalStride = 192;      // FP64 scalar slots per replica

// Partial-sum slots: one array of per-block FP64 partials per slot and replica.  Reducing a
// slot is done redundantly, in a fixed order, by every block that needs the total, so the
// result is bit-identical in all blocks and from run to run.
enum PartSlot {
    P_Q = 0,     // sum_r G_N(r)            (written by the last forward contour step; nq entries)
    P_ES,        // sum_r exp(-U_S)         (written by the Boltzmann-factor kernel)
    P_H0,        // <g, d>
    P_CD,        // <d, phi_m d>
    P_H1,        // <phi* - phi[U + a1 d], d>
    P_GG0,       // <g, g>, even iterations
    P_GG1,       // <g, g>, odd iterations
    P_GMAX,      // max |g|
    P_MASS0, P_MASS1, P_MASS2,   // sum_r phi_I after the convection-diffusion update
    P_RHO, P_JX, P_JY, P_JZ,     // LB mass and momentum
    P_UMAX,      // max |u_lat|
    P_OBS0, P_OBS1, P_OBS2, P_OBS3, P_OBS4, P_OBS5,   // observables (dscf_observables)
    NPART
};

// Scalar history slots (per replica, FP64).
enum ScalSlot {
    S_GG0 = 0, S_GMAX0 = 1,      // start of the inversion
    S_ITER0 = 2,                 // per iteration k: a1, a, gg, gmax at S_ITER0 + 4k + {0..3}
    S_Q = 160, S_QS, S_DRIFT0, S_DRIFT1, S_DRIFT2, S_MASS0, S_MASS1, S_MASS2,
    S_RHO, S_JX, S_JY, S_JZ, S_UMAX, S_PERR,
    S_NITER,                     // inversion iterations run in the last step (residual stop)
    // totals of partial sums, formed once by the last block of the kernel that wrote them:
    S_H0S, S_CDS, S_H1S,         // line search: <g,d>, <d, phi_m d>, h1
    S_GGS0, S_GGS1,              // <g,g> in the parity slots of the iterations
    S_TOT0, S_TOT1, S_TOT2,      // sum_r phi_I before the mass correction
    S_QSUM, S_QLO, S_ESS, S_ESLO,   // sum_r G_N(r) and sum_r exp(-U_S) of the last evaluation (FP64: two parts)
    S_SHF0, S_SHF1, S_SHF2,      // mass correction per site
    S_QFIN,                      // finished-brick count of the sweeps (an unsigned)
    S_WARM,                      // steps whose starting potentials Uprev holds (0, 1, 2 = enough)
    S_FIN = kScalStride - 1      // finished-block count (an unsigned in this slot's bytes)
};

// Device status bits.
enum { ST_NONFINITE = 1, ST_TIMEOUT = 2 };
// Layout of the status block: [0] status word, [1] LB step counter, [2] abort flag of the
// persistent sweeps, [3] change flag of the solvent-component labelling, [kCoopBase..] the barrier
// counters of the general sweeps (three lines), [kFlagBase..] the step counters of the persistent
// bricks.
constexpr int kCoopBase = 32;
constexpr int kFlagBase = 128;
constexpr int kFlagStride = 32;   // ints between bricks' step counters: one 128-byte line each
constexpr int kFlagChain = 16;    // the backward chain's counter in that line (the forward's is first)
constexpr int kMaxBricks = 4096;
// status block: the words above, kMaxBricks counters, then the int4 brick table of the sweeps
constexpr size_t kStatusInts = (size_t)kFlagBase + (size_t)kMaxBricks * kFlagStride + 4 * (size_t)kMaxBricks;

// Parameters of a replica in the field precision, formed on the host.  In the FP32 kernels a thread forms
// none from the FP64 ones: GB300 issues two FP64 lanes a clock and SM, so one conversion or product per
// thread costs as much as 64 FP32 instructions, and a division per thread of a 586-block launch 4 us.
// With these, one thread per block for the rest and the block sums below, a coupled step of six iterations
// at 48^3, N = 16, FP32 fell from 1.29 to 1.02 ms, one of four at 128^3, N = 64 from 4.00 to 3.71 ms.
template <typename T>
struct Par {
    T al, be;                  // stencil: alpha, 1 - 2 alpha
    T rr;                      // the sweeps' passes: c + rr (a + d), rr = alpha / (1 - 2 alpha)
    T ew;                      // weight of the copolymer's Boltzmann factors, near 1 / (1 + 2 rr)^3
    T s1;                      // the three passes of the constant field 1, rounded as the sweeps round it
    double qn;                 // Q from the sweeps' mean of G_N, which holds N weights
    T rho0, gs, gb, dt2;       // LB: density, 1 - 1/tau, dt^2
    T dtM, c, kappa, floor;    // diffusion: dt M, dt M / 2, compressibility, floor of phi
    T chi[9];
    T amp2, kT;                // thermal noise
};

// One replica as the kernels see it.  Pointers are into the caller's workspace; their element
// type is the context precision (double or float) except part/scal (double).
struct Rep {
    int nx, ny, nz, ns, N, nA;
    long long V;
    int nq;                                // P_Q partials to sum in norm_of; 0: scal[S_QSUM] is the total
    int nq_units;                          // general sweeps: row planes, entries of qrow
    int blk0, nblk, chunk;                 // flat tiling: nblk blocks of `chunk` sites
    int lb_blk0, lb_nblk;                  // LB grid: one site per thread, lb_nblk blocks
    int hydro, cn_sweeps;
    double phi_p, kappa, alpha, dt, M, gs, gb, rho0, phi_floor;
    double chi[9];
    double mass0[3];
    Par<float> pf;
    Par<double> pd;
    long long ext_off;                     // offset of this replica in [rep][ns][V] arrays
    long long vbase;                       // sites of the replicas before it ([rep][c][V] arrays)
    void* phi;   // [ns][V] compositions (target of the inversion)
    void* U;     // [ns][V]
    void* mu;    // [ns][V]
    void* d;     // [ns][V] conjugate direction
    void* phim;  // [ns][V] phi[U]
    void* q;     // [2][V]  contour quadratures
    void* E;     // [ns][V] Boltzmann factors exp(-U)
    void* G;     // [N][V]  forward propagators G_1..G_N
    void* Gp0;   // [V]     general sweeps: a chain's first level past the middle, forward
    void* Gp1;   // [V]     and backward; bricks: the backward chain's boundary rows past the middle
    void* u;     // [3][V]  LB velocity (lattice units)
    void* pop0;  // [19][V] LB population deviations (post-collision), even steps
    void* pop1;  // [19][V] odd steps
    void* del0;  // [ns][V] Jacobi iterates; bricks: the forward chain's boundary rows past the middle
    void* del1;  // [ns][V]
    void* rhs;   // [ns][V] right-hand side of the Crank-Nicolson system
    void* Uprev; // [ns][V] potentials the previous step's inversion started from
    // thermal noise (dscf_set_noise): composition flux variance 2 M dt / Omega per unit phi,
    // LB temperature dt^2 / Omega (0: off), generator key
    double noise_amp2, noise_kT;
    unsigned long long noise_seed;
    int rep_index;                         // counter word 3 of the noise (replica in the batch)
    double* qrow;   // general sweeps: sums of G_N per row plane
    double* part;   // [NPART][part_stride]
    int part_stride;
    double* scal;   // [kScalStride]
};

template <typename T>
__host__ __device__ __forceinline__ const Par<T>& pars(const Rep& R) {
    if constexpr (sizeof(T) == 4) return R.pf;
    else return R.pd;
}
// (Re)forms pf and pd from the FP64 parameters.
template <typename T>
inline void set_par(const Rep& R, Par<T>& p) {
    const double be = 1.0 - 2.0 * R.alpha;
    p.al = (T)R.alpha; p.be = (T)be;
    // (FP32: 1 - 2 alpha no smaller than 2^-25, a change of alpha below its own rounding, so that a level grows
    // by at most 2^75 within the passes; alpha may be as close to 1/2 as FP64 holds it, and (1 / be)^3 then
    // passes 1e38)
    p.rr = (T)(R.alpha / (sizeof(T) == 4 && be < 0x1p-25 ? 0x1p-25 : be));
    // The passes leave out their centre weights, so a level grows by w3 = (1 + 2 rr)^3 and the factors carry
    // a weight against it.  Any weight will do (it cancels in the densities); a power of two adds no
    // rounding to the factors, which are the same at every bead of a block: with 1 / w3 the potentials of a
    // 128^3 FP64 step were 3 times as far off.  The nearest power leaves a level a drift of up to sqrt 2, so
    // it is taken only where the whole chain drifts by less than a twelfth of the exponents' range (2^10 in
    // FP32, 2^80 in FP64); other chains take 1 / w3.
    const long double w = 1.0L + 2.0L * (long double)p.rr, w3 = w * w * w;
    const double lw = std::log2((double)w3), drift = R.N * std::fabs(lw - std::round(lw));
    p.ew = drift <= (sizeof(T) == 4 ? 10 : 80) ? (T)std::exp2(-std::round(lw)) : (T)(1.0L / w3);
    const T t = std::fma(p.rr, T(2), T(1)), u = std::fma(p.rr, t + t, t);
    p.s1 = std::fma(p.rr, u + u, u);
    long double qn = w3 / (long double)p.s1, f = 1.0L / ((long double)p.ew * w3);
    for (int n = R.N; n; n >>= 1, f *= f)   // (a call of pow in long double takes some microseconds on the host)
        if (n & 1) qn *= f;
    p.qn = (double)qn;
    p.rho0 = (T)R.rho0; p.gs = (T)R.gs; p.gb = (T)R.gb; p.dt2 = (T)(R.dt * R.dt);
    p.dtM = (T)(R.dt * R.M); p.c = (T)(0.5 * R.dt * R.M); p.kappa = (T)R.kappa; p.floor = (T)R.phi_floor;
    for (int i = 0; i < 9; ++i) p.chi[i] = (T)R.chi[i];
    p.amp2 = (T)R.noise_amp2; p.kT = (T)R.noise_kT;
}
inline void set_pars(Rep& R) {
    set_par(R, R.pf);
    set_par(R, R.pd);
}

// Flat tiling of one replica; the context path and the allocation-free path both use it.
inline void tile_replica(Rep& R) {
    long long nb = (R.V + kFlatThreads - 1) / kFlatThreads;
    if (nb > kMaxFlatBlocks) nb = kMaxFlatBlocks;
    long long chunk = (R.V + nb - 1) / nb;
    chunk = (chunk + kFlatThreads - 1) / kFlatThreads * kFlatThreads;
    R.chunk = (int)chunk;
    R.nblk = (int)((R.V + chunk - 1) / chunk);
    R.lb_nblk = (int)((R.V + kFlatThreads - 1) / kFlatThreads);
}

// Launch description shared by the host launchers.
struct Launch {
    const Rep* reps;         // device table
    const int* blk2rep;      // device map: flat block -> replica
    int* status;             // device status word
    int* counter;            // device step counter (selects the LB buffer parity)
    int nblk_total;          // flat blocks over all replicas
    int nlb_total;           // LB blocks over all replicas
    int nrep;
    int noise;               // thermal noise: 1 compositions, 2 LB modes
    cudaStream_t stream;
};

// ---------------------------------------------------------------------------------------------
// Deterministic reductions (warp shuffle then one warp over the warp sums).
// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ double warp_sum(double v) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}
__device__ __forceinline__ double warp_max(double v) {
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_down_sync(0xffffffffu, v, o));
    return v;
}

// Block-wide sum; the result is returned to every thread.  sh: >= 33 doubles of shared memory.
__device__ __forceinline__ double block_sum(double v, double* sh) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nw = (blockDim.x * blockDim.y + 31) >> 5;
    const int tid = threadIdx.x + threadIdx.y * blockDim.x;
    const int l = tid & 31, w = tid >> 5;
    (void)lane; (void)warp;
    v = warp_sum(v);
    if (l == 0) sh[w] = v;
    __syncthreads();
    if (w == 0) {
        double x = (l < nw) ? sh[l] : 0.0;
        x = warp_sum(x);
        if (l == 0) sh[32] = x;
    }
    __syncthreads();
    double r = sh[32];
    __syncthreads();
    return r;
}

// NV block-wide sums in one pass (same order per value as block_sum, so the same results).
// sh: >= 33 NV doubles of shared memory.
template <int NV>
__device__ __forceinline__ void block_sum_n(double (&v)[NV], double* sh) {
    const int nw = (blockDim.x * blockDim.y + 31) >> 5;
    const int tid = threadIdx.x + threadIdx.y * blockDim.x;
    const int l = tid & 31, w = tid >> 5;
#pragma unroll
    for (int k = 0; k < NV; ++k) {
        v[k] = warp_sum(v[k]);
        if (l == 0) sh[33 * k + w] = v[k];
    }
    __syncthreads();
    if (w == 0) {
#pragma unroll
        for (int k = 0; k < NV; ++k) {
            double x = (l < nw) ? sh[33 * k + l] : 0.0;
            x = warp_sum(x);
            if (l == 0) sh[33 * k + 32] = x;
        }
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < NV; ++k) v[k] = sh[33 * k + 32];
    __syncthreads();
}

// NV block-wide FP64 sums of one value per thread of a kFlatThreads block, in a fixed order, returned to
// thread 0 only.  For FP32 values one warp per sum takes the threads' values from shared memory, eight
// per lane: 13 FP64 warp instructions a sum instead of 53 (every warp shuffling its own).
// sh: NV x 33 doubles.
template <int NV>
__device__ __forceinline__ void block_total(const float (&v)[NV], double* sh, double (&out)[NV]) {
    static_assert(NV <= kFlatThreads / 32 && kFlatThreads * sizeof(float) <= 128 * sizeof(double), "one warp per sum");
    __shared__ float val[NV][kFlatThreads];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < NV; ++k) val[k][threadIdx.x] = v[k];
    __syncthreads();
    if (w < NV) {
        double s = 0.0;
#pragma unroll
        for (int i = 0; i < kFlatThreads / 32; ++i) s += (double)val[w][32 * i + lane];
        s = warp_sum(s);
        if (lane == 0) sh[w] = s;
    }
    __syncthreads();
    if (threadIdx.x == 0)
#pragma unroll
        for (int k = 0; k < NV; ++k) out[k] = sh[k];
}
template <int NV>
__device__ __forceinline__ void block_total(const double (&v)[NV], double* sh, double (&out)[NV]) {
#pragma unroll
    for (int k = 0; k < NV; ++k) out[k] = v[k];
    block_sum_n<NV>(out, sh);
}
// Block-wide maximum, returned to thread 0 (FP32 values are compared as such).
__device__ __forceinline__ double block_top(float v, double* sh) {
    float* f = (float*)sh;
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_down_sync(0xffffffffu, v, o));
    __syncthreads();
    if ((threadIdx.x & 31) == 0) f[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0)
        for (int i = 1; i < kFlatThreads / 32; ++i) v = fmaxf(v, f[i]);
    return (double)v;
}

__device__ __forceinline__ double block_max(double v, double* sh) {
    const int nw = (blockDim.x * blockDim.y + 31) >> 5;
    const int tid = threadIdx.x + threadIdx.y * blockDim.x;
    const int l = tid & 31, w = tid >> 5;
    v = warp_max(v);
    if (l == 0) sh[w] = v;
    __syncthreads();
    if (w == 0) {
        double x = (l < nw) ? sh[l] : 0.0;
        x = warp_max(x);
        if (l == 0) sh[32] = x;
    }
    __syncthreads();
    double r = sh[32];
    __syncthreads();
    return r;
}

__device__ __forceinline__ double block_top(double v, double* sh) { return block_max(v, sh); }

// A sum carried with its rounding errors (Knuth's two-sum).  The totals of Q and of exp(-U_S) in FP64 end in
// a few additions of numbers as large as themselves, whose roundings nothing averages out: up to 2e-16 of
// the total and so of every density.
struct Two {
    double hi, lo;
};
__device__ __forceinline__ Two operator+(const Two& a, const Two& b) {
    const double s = a.hi + b.hi, z = s - a.hi;
    return {s, ((a.hi - (s - z)) + (b.hi - z)) + (a.lo + b.lo)};
}
__device__ __forceinline__ Two warp_sum(Two v) {   // in every lane
    for (int o = 16; o > 0; o >>= 1)
        v = v + Two{__shfl_xor_sync(0xffffffffu, v.hi, o), __shfl_xor_sync(0xffffffffu, v.lo, o)};
    return v;
}
// Total of n partials read through L2, by a warp.  Only the last additions carry their errors: a lane's own
// are of parts of the total, and their roundings average out.
__device__ __forceinline__ Two total_of(const double* p, int n) {
    double s = 0.0;
    for (int i = threadIdx.x & 31; i < n; i += 32) s += __ldcg(p + i);
    return warp_sum(Two{s, 0.0});
}

// Total of n partials, same fixed order in every block.
__device__ __forceinline__ double reduce_parts(const double* __restrict__ p, int n, double* sh) {
    const int tid = threadIdx.x + threadIdx.y * blockDim.x;
    const int nt = blockDim.x * blockDim.y;
    double s = 0.0;
    for (int i = tid; i < n; i += nt) s += p[i];
    return block_sum(s, sh);
}
// Totals of NV partial arrays of n entries each, in one pass (same results as reduce_parts).
template <int NV>
struct Parts {
    const double* p[NV];
};
template <int NV>
__device__ __forceinline__ void reduce_parts_n(const Parts<NV> p, int n, double (&out)[NV], double* sh) {
    const int tid = threadIdx.x + threadIdx.y * blockDim.x;
    const int nt = blockDim.x * blockDim.y;
#pragma unroll
    for (int k = 0; k < NV; ++k) out[k] = 0.0;
    for (int i = tid; i < n; i += nt)
#pragma unroll
        for (int k = 0; k < NV; ++k) out[k] += p.p[k][i];
    block_sum_n<NV>(out, sh);
}
// The same totals read through L2 (ld.global.cg), for partials that other blocks of the running
// kernel have just written.
__device__ __forceinline__ double reduce_parts_cg(const double* p, int n, double* sh) {
    const int tid = threadIdx.x + threadIdx.y * blockDim.x;
    const int nt = blockDim.x * blockDim.y;
    double s = 0.0;
    for (int i = tid; i < n; i += nt) s += __ldcg(p + i);
    return block_sum(s, sh);
}
template <int NV>
__device__ __forceinline__ void reduce_parts_n_cg(const Parts<NV> p, int n, double (&out)[NV], double* sh) {
    const int tid = threadIdx.x + threadIdx.y * blockDim.x;
    const int nt = blockDim.x * blockDim.y;
#pragma unroll
    for (int k = 0; k < NV; ++k) out[k] = 0.0;
    for (int i = tid; i < n; i += nt)
#pragma unroll
        for (int k = 0; k < NV; ++k) out[k] += __ldcg(p.p[k] + i);
    block_sum_n<NV>(out, sh);
}
__device__ __forceinline__ double reduce_parts_max(const double* __restrict__ p, int n, double* sh) {
    const int tid = threadIdx.x + threadIdx.y * blockDim.x;
    const int nt = blockDim.x * blockDim.y;
    double s = 0.0;
    for (int i = tid; i < n; i += nt) s = fmax(s, p[i]);
    return block_max(s, sh);
}

__device__ __forceinline__ double* slot(const Rep& R, int s) { return R.part + (size_t)s * R.part_stride; }

// Fence-and-count: after thread 0 of every block of the replica has written its partials, true in
// the one block that finishes last, where every block's partials are visible.  The count wraps
// to zero at R.nblk, so it is ready for the next launch without a reset.  The last block forms
// the totals once (in the same order as reduce_parts), instead of every block of the consuming
// kernel re-reading all partials of one L2 line set.
__device__ __forceinline__ bool last_block_of(const Rep& R, int* flag_sh) {
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        const unsigned old = atomicInc((unsigned*)(R.scal + S_FIN), (unsigned)R.nblk - 1u);
        *flag_sh = (old == (unsigned)R.nblk - 1u);
    }
    __syncthreads();
    const bool last = *flag_sh != 0;
    if (last) __threadfence();
    return last;
}

// Waits of the contour sweeps: acquire loads of other CTAs' counters, mbarriers in shared memory.
__device__ __forceinline__ unsigned saddr(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ int ld_acquire(const int* p) {
    int v;
    asm volatile("ld.acquire.gpu.global.s32 %0, [%1];\n" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void bar_init(unsigned long long* bar, int count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(saddr(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void bar_arrive(unsigned long long* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(saddr(bar)) : "memory");
}
__device__ __forceinline__ bool bar_test(unsigned long long* bar, unsigned parity) {
    unsigned done;
    asm volatile(
        "{\n\t.reg .pred P1;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 P1, [%1], %2;\n\t"
        "selp.b32 %0, 1, 0, P1;\n\t}\n"
        : "=r"(done)
        : "r"(saddr(bar)), "r"(parity)
        : "memory");
    return done != 0;
}
// Polls of a shared-memory mbarrier before giving up.  What completes them (a CTA's own copies, its compute
// warps, its exchange or barrier warps, whose waits on other CTAs are bounded by the context's limit)
// depends on no unbounded wait, so this bound is fixed and far above any real time (a shorter limit set for
// failure tests must not abandon a copy that is still landing in this CTA's shared memory).
constexpr long long kBarSpinLimit = 1LL << 28;

// Boltzmann factor exp(-x) in the field precision (CUDA's exp / expf, not re-implemented).
// Philox4x32-10 (Salmon, Moraes, Dror, Shaw, SC'11): ten rounds; each multiplies counter words 0
// and 2 by 0xD2511F53 and 0xCD9E8D57 (32 x 32 -> 64 bits), XORs the high halves into words 1 and
// 3 with the key, and swaps; the key advances by the Weyl constants 0x9E3779B9, 0xBB67AE85.
__device__ __forceinline__ uint4 philox4x32_10(uint4 c, unsigned k0, unsigned k1) {
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        if (r > 0) { k0 += 0x9E3779B9u; k1 += 0xBB67AE85u; }
        const unsigned lo0 = 0xD2511F53u * c.x, hi0 = __umulhi(0xD2511F53u, c.x);
        const unsigned lo1 = 0xCD9E8D57u * c.z, hi1 = __umulhi(0xCD9E8D57u, c.z);
        c = make_uint4(hi1 ^ c.y ^ k0, lo1, hi0 ^ c.w ^ k1, lo0);
    }
    return c;
}
// Four standard normals of counter (site, step, stream, replica): uniforms (top 24 bits + 1/2) /
// 2^24, Box-Muller on words (0, 1) and (2, 3).
template <typename T>
__device__ __forceinline__ void normals4(unsigned long long seed, unsigned site, unsigned step, unsigned stream,
                                         unsigned rep, T (&n)[4]) {
    const uint4 r = philox4x32_10(make_uint4(site, step, stream, rep), (unsigned)seed, (unsigned)(seed >> 32));
    const unsigned w[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
    for (int pr = 0; pr < 2; ++pr) {
        const T ua = ((T)(w[2 * pr] >> 8) + T(0.5)) * T(1.0 / 16777216.0);
        const T ub = ((T)(w[2 * pr + 1] >> 8) + T(0.5)) * T(1.0 / 16777216.0);
        T sn, cs;
        if constexpr (sizeof(T) == 4) {
            const float rad = sqrtf(-2.f * logf(ua));
            sincospif(2.f * ub, &sn, &cs);
            n[2 * pr] = rad * cs;
            n[2 * pr + 1] = rad * sn;
        } else {
            const double rad = sqrt(-2.0 * log(ua));
            sincospi(2.0 * ub, &sn, &cs);
            n[2 * pr] = rad * cs;
            n[2 * pr + 1] = rad * sn;
        }
    }
}

__device__ __forceinline__ double bexp(double x) { return exp(-x); }
__device__ __forceinline__ float bexp(float x) { return expf(-x); }

// ---------------------------------------------------------------------------------------------
// Host launchers (defined in the kernel translation units, explicit per precision).
// ---------------------------------------------------------------------------------------------
// General sweeps of both chains (dscf_coop.cuh), levels j0 .. j1 - 1: a cooperative launch for several
// levels, a plain one for one.  kk: row layout of every replica, 0 if they differ.
// A replica as the general sweeps see it; their table holds the replicas by decreasing chain length.  (120
// bytes: with 128 the kernel's table would pass 16 KB of shared memory, whose next size takes 16 KB from the
// L1 cache; 256^3, N = 64: 7.43 and 7.51 ms.)
struct CoopRep {
    int nx, ny, nz, N, nA;
    short layout;        // coop_layout
    short strip;         // rows cut together: 8 (a CTA's warps side by side) or 1
    int units;           // row planes
    int tile;            // sites of an x tile (coop_tile); mode 4: rows of a group
    int wgt, cost0;      // cost of a plane of a strip, of all entries before
    long long V;
    void *E, *G, *Gp0, *Gp1, *q;
    double *qrow, *pq;   // sums of G_N per row plane (or nullptr), the P_Q slot
    double* qsum;        // where their total goes
    double rr;           // Par<T>::rr
};
static_assert(sizeof(CoopRep) <= 120, "the general sweeps' table");
struct CoopPlan {
    const CoopRep* reps; // device table
    int nrep;
    int* cnt;            // device: barrier counters (3 lines), zero between launches
    int* abort;
    int kk, ncta;
    int runs, per;       // runs > 0: one replica, each row cut into this many, one per warp, `per` in a CTA
};
// Row layout of a grid: sites per lane + 16 (1 + mode), mode 0 blocked, 1 strided, 2 and 3 the same in x
// tiles (rows of more than 256 sites).  Blocked for the smallest K of 1, 2, 3, 4, 6, 8 that divides nx into
// at most 32 lanes, up to one and a half times what 32 full lanes would need.
constexpr int kCoopRow = 256;   // longest untiled row
// Tiles of a longer row: of up to 30 groups of 4 sites where they divide it, else of up to 126 or 158 sites
// (4 or 5 a lane, the fewer lanes in all; 6 a lane lose: 511 x 255 x 63 FP32), two lanes or columns more
// being the neighbours' on either side (coop_run).
__host__ __device__ constexpr int coop_tile_k(int nx) {   // sites per lane
    return nx % 4 == 0 || 4 * ((nx + 125) / 126) <= 5 * ((nx + 157) / 158) ? 4 : 5;
}
__host__ __device__ constexpr int coop_tiles(int nx) {
    return nx <= kCoopRow ? 1 : nx % 4 == 0 ? (nx / 4 + 29) / 30 : coop_tile_k(nx) == 4 ? (nx + 125) / 126 : (nx + 157) / 158;
}
__host__ __device__ constexpr int coop_tile(int nx) {   // sites of a tile; the last may have fewer
    const int t = coop_tiles(nx), u = nx <= kCoopRow || nx % 4 ? 1 : 4;
    return u * ((nx / u + t - 1) / t);
}
// Short rows of FP32 fields that hold many of them: a warp takes as many adjacent rows as its lanes hold, with
// 4 or 2 sites a lane, mode 4.  One row a warp has a quarter of the bytes in flight or less; small fields,
// whose rows are to fill all warps, take one, and FP64, bound by its pipe.  Density evaluations, N = 24, us, one
// row a warp and groups: 16^3 100, 110; 32^3 103, 110; 32 x 64 x 64 122, 119; 24 x 100 x 100 160, 136; 16 x 128 x
// 128 198, 131; 32 x 512 x 512 2662, 1541 (a launch per level, before these sweeps: 2433); 24 x 600 x 600 3636,
// 1667 (3087); 8 x 1000 x 1000 8365, 1498 (7384).
__host__ __device__ constexpr bool coop_narrow(int nx, long long V, bool fp64) {
    return !fp64 && nx <= 32 && nx % 2 == 0 && V >= (1LL << 17);
}
__host__ __device__ constexpr int coop_group(int nx, long long V, bool fp64) {   // rows of a warp
    return coop_narrow(nx, V, fp64) ? 32 / (nx / (nx % 4 == 0 ? 4 : 2)) : 1;
}
__host__ __device__ constexpr int coop_layout(int nx, long long V, bool fp64) {
    if (coop_narrow(nx, V, fp64)) return (nx % 4 == 0 ? 4 : 2) + 80;
    if (nx > kCoopRow) return coop_tile_k(nx) + (nx % 4 == 0 ? 64 : 48);
    const int k = (nx + 31) / 32;
    for (int K = k; K <= 8 && 2 * K <= 3 * k + 1; ++K)
        if (K != 5 && K != 7 && nx % K == 0) return K + 16;
    return k + 32;
}
// Compute warps of a CTA of the general sweeps (kk: the row layout of all replicas, or 0).
__host__ __device__ constexpr int coop_warps(int kk, bool fp64) { return kk > 0 && (kk & 15) * (fp64 ? 8 : 4) <= (fp64 ? 16 : 24) ? 12 : 8; }
constexpr int kCoopMaxCtas = 152;
long long coop_units(const Rep& R, bool fp64);   // planes of rows, of x tiles or of groups of rows
int coop_cost(const Rep& R, bool fp64);   // of a row plane
void coop_cut(CoopPlan& c, const Rep& R, long long work, bool fp64, int nsm);   // ncta, runs, per
CoopRep coop_rep(const Rep& R, bool fp64, int cost, int cost0);   // cost: of a row plane
template <typename T> const void* coop_mixed();   // the kernel of replicas of unlike row layouts
template <typename T> int coop_prepare(int kk);   // cudaError_t
template <typename T> int launch_prop_coop(const Launch& L, const CoopPlan& c, int j0, int j1, int limit);   // cudaError_t
// mode: 0 exp(-U), 1 trial exp(-(U + a1 d)), 2 commit U += a d then exp(-U), 3 exp(-Uext)
template <typename T> void launch_exp(const Launch& L, int mode, int k, const void* Uext, int write_u = 0);
// net != 0: the density at the evaluated potential is the learned predictor's output, stored in q
template <typename T> void launch_trial(const Launch& L, int net = 0);
template <typename T> void launch_grad(const Launch& L, int k, int net = 0);
// Residual stop of the inversion before iteration k: sets the graph condition `handle` to 1 while
// max|g| >= tol for some replica (0 otherwise, also for a non-finite residual) and records the
// iterations run in scal[S_NITER]; k = 0 also records the start-of-inversion residual.
void launch_ncg_gate(const Launch& L, int k, double tol, unsigned long long handle);
void launch_pred_err(const Launch& L);   // max |q - phi_m| of replica 0 into scal[S_PERR] (FP32 melts)
// Observables: pass 1 leaves per-block sums of phi_I (slots P_OBS0..2), U.phi (P_OBS3) and the
// interaction energy density (P_OBS4); pass 2, given the species means, sum (phi_I - <phi_I>)^2
// over I (P_OBS0) and |phi_A + phi_B - <phi_A> - <phi_B>| (P_OBS1).
template <typename T>
void launch_obs1(const Launch& L);
template <typename T>
void launch_obs2(const Launch& L, double mA, double mB, double mS);
// per-block counts of cubes, faces, edges, vertices of {phi_species > threshold} into P_OBS0..3
template <typename T> void launch_minkowski(const Launch& L, int replica, int species, double threshold);
// trapped solvent: component labels of the complement of {phi_B > threshold} (lab, cnt: V ints)
template <typename T> void launch_cc_init(const Launch& L, int replica, double threshold, int* lab, int* cnt);
void launch_cc_step(const Launch& L, int replica, int* lab, int* changed);
void launch_cc_count(const Launch& L, int replica, const int* lab, int* cnt);   // P_OBS0/1 largest size/root, P_OBS4 roots
template <typename T> void launch_cc_solvent(const Launch& L, int replica, const int* lab, int bulk);   // P_OBS2, 3
// mode 0: init (d = -g), mode 1: iteration k direction update
template <typename T> void launch_dir(const Launch& L, int mode, int k);
template <typename T> void launch_mu(const Launch& L, int K);   // K < 0: iterations from scal[S_NITER]
template <typename T> void launch_extrap(const Launch& L);       // extrapolated start of the inversion
template <typename T> void launch_lb(const Launch& L, const void* force_ext);
template <typename T> void launch_cd(const Launch& L, int sweeps);
template <typename T> void launch_dens_out(const Launch& L, void* phi_ext);
template <typename T> void launch_pop_copy(const Launch& L, void* ext, int dir);  // 0 get, 1 set
template <typename T> void launch_mass_init(const Launch& L, int nrep);
void launch_step_end(const Launch& L);
template <typename T> void launch_lb_diag(const Launch& L);
// persistent contour sweeps (FP32; row widths 32, 48, 64, 96, 128; several replicas of one width
// per launch, each CTA taking its brick from an int4 table: replica, brick in the replica, flag
// index of the replica's brick 0)
// Brick rows: 16 for rows of at most 64 sites (so that a brick, and the co-resident launch, holds
// as many sites as for the wider rows) where ny allows it, else 8.
__host__ __device__ inline int pers_pby_of(int nx, int ny) { return (nx <= 64 && ny % 16 == 0) ? 16 : 8; }
size_t pers_smem_bytes(int width, int pby, int bz);
size_t pers_mix_smem_bytes(int bz);                            // the mixed-width launches (width 0)
bool pers_width_ok(int nx);
int pers_pby(const Rep& R);                                    // brick rows of a replica (8 or 16)
bool pers_supported(const Rep& R, int bz, int nw, int nsm);   // nw: warps per CTA
int pers_bricks(const Rep& R, int bz);   // the uppermost may have fewer planes
// width 0: bricks of several widths in one launch; rag (16 planes, one width): fewer planes in the uppermost
int pers_prepare(int width, int pby, int bz, int nw, bool rag);   // cudaError_t
int launch_prop_pers(const Launch& L, int width, int pby, int bz, int nw, bool rag, int nbricks, const int4* table,
                     int* flags, int* abortf, int limit);  // cudaError_t
// SM id of each CTA of a sweep-shaped cooperative launch (cudaError_t)
int pers_placement(int bz, int nw, int nbricks, int* d_smid, cudaStream_t stream);

}  // namespace dscf

namespace dscf {
// tcgen05 forward convolution of the predictor network (dscf_tc.cu)
bool tc_conv_supported(int nx, int ny);
size_t tc_conv_smem();
int tc_conv_prepare();   // cudaError_t
int tc_conv_blocks(int nx, int ny, int nz);   // CTAs per sample
void launch_conv_tc(int layer, const void* in, const void* wt, const float* bias, int cout, void* out, int nx, int ny,
                    int nz, int B, double* part, int* err, cudaStream_t s);
}  // namespace dscf
// learned predictor (dscf_net.cu): forward pass on a given stream, for use inside the step graph
struct dscf_net;
bool dscf_net_fits(const dscf_net* net, int nx, int ny, int nz);
int dscf_net_forward_launches(const dscf_net* n);   // kernels one forward pass launches
void dscf_net_forward_on(dscf_net* net, cudaStream_t stream, const float* U, double pb0, double pb1, float* phi);
