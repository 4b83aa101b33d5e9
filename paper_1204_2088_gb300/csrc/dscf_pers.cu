// Persistent contour sweeps (Eq. 16-17) in the whole-row layout (FP32), for one replica or a
// batch of replicas.
//
// One launch runs both chains of a density evaluation: the forward propagator G_s (s = 1 .. N) and
// the backward one G+_s (s = N .. 1) do not depend on each other until the quadrature, so every
// CTA advances them in turn, one contour step of each (a "unit") at a time, and they meet in the
// middle, h = ceil(N / 2): the forward chain stores G_s for s <= h and the backward chain G+_s for
// s > h in the contour stack; past the middle each chain multiplies sigma of its own field with the
// stored value of the other, q_{I_s} += sigma[G_{s-1}] G+_s = G_s sigma[G+_{s+1}].  The HBM bytes
// are those of one chain after the other (each stack level written once and read once, and the
// levels near the middle are read back while still in L2), but a chain's halo exchange (release,
// neighbours' counters, copies: L2 round trips of 5 to 6 thousand cycles) runs while the SM
// computes the other chain's unit.  128^3, N = 64: 540 us for the two sweeps one after the other
// (4.2 us a contour step, the exchange in the open), 362 us so (2.8 us).
//
// The lattice is cut into bricks of nx x PBY x BZ sites, one brick per CTA and one CTA per SM (the
// launch is cooperative, so all CTAs are resident together), one compute warp per plane of the
// brick and four warps for the exchange.  Rows of 96 or 128 sites
// are held by a whole warp (3 or 4 sites per lane), rows of 32, 48 or 64 sites by half a warp (2,
// 3 or 4 sites per lane), two rows side by side; bricks of these narrow rows have 16 rows instead
// of 8 where ny allows it.  A CTA takes its brick from a table (replica, brick, flag base), so
// replicas share a launch; a brick waits only on the bricks of its own replica.
//
// Per unit a compute warp
//   takes the halo rows of the previous step from shared memory (x pass in registers), y-filters
//   its plane in registers (the x-filtered rows of both chains stay in registers from step to
//   step) into shared YS, and one row of a z-halo plane;
//   barrier; z pass (the neighbouring planes from YS), times the Boltzmann factor; boundary stores
//   and, past the middle, the quadrature; arrives on the unit's `pub` mbarrier;
//   stores the interior of a stack level or fetches the next unit's one; x pass in registers.
// The exchange warps (two per chain) wait for `pub`, publish the brick's step counter of that chain
// with a release store, wait for its eight y/z neighbours' counters and copy the next step's raw
// halo rows into shared memory (cp.async, completing on the chain's `full` mbarrier).  `pub` is also
// what keeps YS from being overwritten before every warp's z pass has read it, so a unit has one
// CTA barrier.
//
// The Boltzmann factors of both species and both quadrature accumulators (each as large as the
// brick) live in tensor memory, one 32-bit column per thread and value (tcgen05.ld / st): beside
// the two chains' rows they do not fit in the registers.  The allocation never waits for another
// sweep: the registers let one CTA of 16 compute warps (all 512 columns) or one of 8 (256) on an
// SM, whatever context or stream they belong to.
// Each 1-D pass of the separable stencil is one add and one fma per site, as packed f32x2 pairs
// (a scalar tail for three sites per lane), with the centre weight left out and made up for by the
// Boltzmann factors.  Every wait is bounded: on timeout the CTA sets a status bit and a global abort flag
// that makes every other CTA stop waiting, so the launch always finishes.
#include "dscf_internal.cuh"

#include <algorithm>
#include <type_traits>

namespace dscf {

namespace {

// Compute warps per CTA: 16 for bricks of 16 planes, 8 for bricks of 8 planes; one CTA per SM.
// Beside them one warpgroup of four warps does the exchange (two per chain): a whole warpgroup, so that
// it can hand most of its registers to the compute warps (setmaxnreg).  Launched registers a thread
// (what the launch bounds leave): 96 for 640 threads, 168 for 384; the shares 512 x 112 + 128 x 32 =
// 640 x 96 and 256 x 208 + 128 x 24 <= 384 x 168 stay within them.
constexpr int kXWarps = 4;
template <int NW>
struct PersRegs {
    static constexpr int compute = NW == 16 ? 112 : 208;
    static constexpr int exchange = NW == 16 ? 32 : 24;
};

__device__ __forceinline__ void cp16(void* s, const void* g) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(saddr(s)), "l"(g));
}
template <int VEC>
__device__ __forceinline__ void cpv(float* s, const float* g) {   // VEC values of a lane: 16, 8 or 3 x 4 bytes
    if constexpr (VEC == 4) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(saddr(s)), "l"(g));
    else if constexpr (VEC == 2) asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(saddr(s)), "l"(g));
    else
#pragma unroll
        for (int k = 0; k < VEC; ++k) asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(saddr(s + k)), "l"(g + k));
}
__device__ __forceinline__ void cp_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }
// arrive on bar (one of its expected arrivals) when all earlier cp.async of this thread have landed
__device__ __forceinline__ void cp_arrive(unsigned long long* bar) {
    asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];\n" ::"r"(saddr(bar)) : "memory");
}
__device__ __forceinline__ void st_release(int* p, int v) {
    asm volatile("st.release.gpu.global.s32 [%0], %1;\n" ::"l"(p), "r"(v) : "memory");
}

// Packed FP32 pairs (sm_100+ f32x2 arithmetic): two lanes of a float4 per instruction.
__device__ __forceinline__ unsigned long long pk2(float a, float b) {
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void upk2(unsigned long long v, float& a, float& b) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ unsigned long long add2(unsigned long long a, unsigned long long b) {
    unsigned long long r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ unsigned long long mul2(unsigned long long a, unsigned long long b) {
    unsigned long long r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ unsigned long long fma2(unsigned long long a, unsigned long long b, unsigned long long c) {
    unsigned long long r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

// Tensor memory: N (2 or 4) consecutive 32-bit columns of the warp's 32 lanes, one lane per thread.
// A load's values are valid after the wait that names them (which also keeps their uses behind it).
template <int N>
__device__ __forceinline__ void tm_ld(unsigned a, float (&v)[N]) {
    if constexpr (N == 4)
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];\n"
                     : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3])
                     : "r"(a));
    else
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x2.b32 {%0, %1}, [%2];\n" : "=f"(v[0]), "=f"(v[1]) : "r"(a));
}
template <int N>
__device__ __forceinline__ void tm_wait_ld(float (&v)[N], float (&u)[N]) {
    if constexpr (N == 4)
        asm volatile("tcgen05.wait::ld.sync.aligned;\n"
                     : "+f"(v[0]), "+f"(v[1]), "+f"(v[2]), "+f"(v[3]), "+f"(u[0]), "+f"(u[1]), "+f"(u[2]), "+f"(u[3]));
    else
        asm volatile("tcgen05.wait::ld.sync.aligned;\n" : "+f"(v[0]), "+f"(v[1]), "+f"(u[0]), "+f"(u[1]));
}
template <int N>
__device__ __forceinline__ void tm_wait_ld(float (&v)[N]) {
    if constexpr (N == 4)
        asm volatile("tcgen05.wait::ld.sync.aligned;\n" : "+f"(v[0]), "+f"(v[1]), "+f"(v[2]), "+f"(v[3]));
    else
        asm volatile("tcgen05.wait::ld.sync.aligned;\n" : "+f"(v[0]), "+f"(v[1]));
}
template <int N>
__device__ __forceinline__ void tm_st(unsigned a, const float (&v)[N]) {
    if constexpr (N == 4)
        asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1, %2, %3, %4};\n" ::"r"(a), "f"(v[0]), "f"(v[1]),
                     "f"(v[2]), "f"(v[3]));
    else
        asm volatile("tcgen05.st.sync.aligned.32x32b.x2.b32 [%0], {%1, %2};\n" ::"r"(a), "f"(v[0]), "f"(v[1]));
}
__device__ __forceinline__ void tm_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;\n" ::: "memory"); }

template <int N>
__device__ __forceinline__ void regs_inc() { asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;\n" ::"n"(N)); }
template <int N>
__device__ __forceinline__ void regs_dec() { asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;\n" ::"n"(N)); }
// Barrier of the compute warps.
__device__ __forceinline__ void compute_sync(int threads) {
    asm volatile("bar.sync 1, %0;\n" ::"r"(threads) : "memory");
}

struct PersCtl {
    int* flags;          // two step counters (chains) per brick, kFlagStride ints apart
    int* abort;          // set by a CTA that gave up waiting
    int* status;         // device status word
    const int4* table;   // per CTA: replica, brick in the replica, flag index of the replica's brick 0
    int limit;           // polls before giving up
};

// Row geometry of a brick of width W and PBY rows: a row is held by LPR lanes, VEC consecutive
// sites each; a warp holds HALVES rows side by side (lanes 0..LPR-1 the first, LPR..31 the
// second), so each lane carries RPL of the plane's PBY rows (rows h RPL .. h RPL + RPL - 1 for
// lane half h).
template <int W, int PBY>
struct PRow {
    static constexpr int LPR = (W == 96 || W == 128) ? 32 : 16;
    static constexpr int VEC = W / LPR;
    static constexpr int HALVES = 32 / LPR;
    static constexpr int RPL = PBY / HALVES;
    static_assert(LPR * VEC == W && VEC >= 2 && VEC <= 4, "row width");
};

// VEC consecutive FP32 values: one vector access for 2 and 4, three scalar ones for 3
template <int VEC>
__device__ __forceinline__ void ldv(const float* p, float (&v)[VEC]) {
    if constexpr (VEC == 4) {
        const float4 t = *(const float4*)p;
        v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
    } else if constexpr (VEC == 2) {
        const float2 t = *(const float2*)p;
        v[0] = t.x; v[1] = t.y;
    } else {
#pragma unroll
        for (int k = 0; k < VEC; ++k) v[k] = p[k];
    }
}
template <int VEC>
__device__ __forceinline__ void stv(float* p, const float (&v)[VEC]) {
    if constexpr (VEC == 4) {
        *(float4*)p = make_float4(v[0], v[1], v[2], v[3]);
    } else if constexpr (VEC == 2) {
        *(float2*)p = make_float2(v[0], v[1]);
    } else {
#pragma unroll
        for (int k = 0; k < VEC; ++k) p[k] = v[k];
    }
}
// Global stores as asm without a memory clobber: the compiler may move the shared-memory loads of the
// next rows over them (it cannot tell that they do not alias).
template <int VEC>
__device__ __forceinline__ void stg(float* p, const float (&v)[VEC]) {
    if constexpr (VEC == 4)
        asm volatile("st.global.v4.f32 [%0], {%1, %2, %3, %4};\n" ::"l"(p), "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]));
    else if constexpr (VEC == 2)
        asm volatile("st.global.v2.f32 [%0], {%1, %2};\n" ::"l"(p), "f"(v[0]), "f"(v[1]));
    else
#pragma unroll
        for (int k = 0; k < VEC; ++k) asm volatile("st.global.f32 [%0], %1;\n" ::"l"(p + k), "f"(v[k]));
}
// o = c + r (a + d) per site: packed pairs, a scalar tail for odd VEC (same rounding: one add, one
// fma per site either way)
template <int VEC>
__device__ __forceinline__ void mixv(const float (&a)[VEC], const float (&c)[VEC], const float (&d)[VEC], float rr,
                                     unsigned long long rr2, float (&o)[VEC]) {
#pragma unroll
    for (int k = 0; k + 1 < VEC; k += 2)
        upk2(fma2(rr2, add2(pk2(a[k], a[k + 1]), pk2(d[k], d[k + 1])), pk2(c[k], c[k + 1])), o[k], o[k + 1]);
    if constexpr (VEC & 1) o[VEC - 1] = __fmaf_rn(rr, __fadd_rn(a[VEC - 1], d[VEC - 1]), c[VEC - 1]);
}
// o = s * v per site
template <int VEC>
__device__ __forceinline__ void mulv(const float (&s)[VEC], const float (&v)[VEC], float (&o)[VEC]) {
#pragma unroll
    for (int k = 0; k + 1 < VEC; k += 2) upk2(mul2(pk2(s[k], s[k + 1]), pk2(v[k], v[k + 1])), o[k], o[k + 1]);
    if constexpr (VEC & 1) o[VEC - 1] = __fmul_rn(s[VEC - 1], v[VEC - 1]);
}
// q += g * v per site
template <int VEC>
__device__ __forceinline__ void fmav(const float (&g)[VEC], const float (&v)[VEC], float (&q)[VEC]) {
#pragma unroll
    for (int k = 0; k + 1 < VEC; k += 2)
        upk2(fma2(pk2(g[k], g[k + 1]), pk2(v[k], v[k + 1]), pk2(q[k], q[k + 1])), q[k], q[k + 1]);
    if constexpr (VEC & 1) q[VEC - 1] = __fmaf_rn(g[VEC - 1], v[VEC - 1], q[VEC - 1]);
}


// Arrays of a replica as the sweep uses them, in shared memory (the descriptor itself is in device
// memory, whose cached copy the acquire loads keep invalidating).
struct PersArrays {
    float* exch[2][2];   // exchange buffers per chain
    float* stack;
    size_t V;
};

// What a compute warp keeps through the sweep.
struct PersWarp {
    const PersArrays& A;
    const PersCtl& ctl;
    unsigned long long *full, *pub;
    float *YS, *HS, *GS;   // GS: the lane's first value of the stack level
    size_t own;            // lane's first site of its first row in a field
    size_t slab;           // lane's 128-byte line of the plane's run in a field (past its end: none)
    int N, nA, hm, w, lane, hf, xo, lsrc, rsrc;
    int planes;            // of the brick
    bool act;              // the warp has one of them
    bool face_plane;
    float rr;
    unsigned long long rr2;
    unsigned tbase;
    float qsum;
    bool dead;
};

// Level j of chain C (contour step s = j + 1 forward, s = N - j backward): the contour stack before
// the chains meet, the chain's exchange buffers (boundary rows only) past it.
__device__ __forceinline__ float* level_of(const PersArrays& A, int c, int N, int hm, int j) {
    return (c ? j < N - hm : j < hm) ? A.stack + (size_t)(c ? N - j - 1 : j) * A.V : A.exch[c][j & 1];
}

// Bounded wait on an mbarrier phase; a thread that gives up reports it and waits no more.
__device__ __forceinline__ void bar_wait(unsigned long long* bar, unsigned parity, const PersCtl& ctl, bool& dead) {
    if (dead) return;
    for (long long spins = 0; !bar_test(bar, parity); ++spins)
        if (spins > kBarSpinLimit) {
            atomicOr(ctl.status, (int)ST_TIMEOUT);
            atomicExch(ctl.abort, 1);
            dead = true;
            return;
        }
}

// x pass of a periodic row: v + r (left + right)
template <int VEC>
__device__ __forceinline__ void xpassv(const PersWarp& k, const float (&v)[VEC], float (&o)[VEC]) {
    const float lv = __shfl_sync(0xffffffffu, v[VEC - 1], k.lsrc);
    const float rv = __shfl_sync(0xffffffffu, v[0], k.rsrc);
    float a[VEC], d[VEC];
#pragma unroll
    for (int i = 0; i < VEC; ++i) {
        a[i] = i ? v[i - 1] : lv;
        d[i] = (i + 1 < VEC) ? v[i + 1] : rv;
    }
    mixv<VEC>(a, v, d, k.rr, k.rr2, o);
}

// Halo rows (row r, plane pl of the brick's frame, r in -1..PBY, pl in -1..BZ) in HS: rows -1, then rows
// 0..PBY-1 of plane -1; rows PBY of planes -1..BZ, then rows 0..PBY-1 of plane BZ.
template <int PBY, int BZ>
__device__ __forceinline__ int halo_row(int r, int pl) {
    constexpr int P = BZ + 2 + PBY;
    if (r < 0) return pl + 1;
    if (r >= PBY) return P + pl + 1;
    return (pl < 0 ? BZ + 2 : P + BZ + 2) + r;
}

// One unit: contour step j of chain C (0 forward, s = j + 1; 1 backward, s = N - j).
template <int W, int PBY, int BZ, int NW, bool RAG, int C>
__device__ __forceinline__ void pers_unit(PersWarp& k, float (&xf)[PRow<W, PBY>::RPL][PRow<W, PBY>::VEC], const int j) {
    using RG = PRow<W, PBY>;
    constexpr int VEC = RG::VEC, LPR = RG::LPR, RPL = RG::RPL;
    constexpr int VS = VEC == 3 ? 4 : VEC;   // tensor-memory columns of a row's sites
    constexpr int NH = 2 * (BZ + 2 + PBY);
    const int N = k.N, hm = k.hm, w = k.w, xo = k.xo;
    const float rr = k.rr;
    const unsigned long long rr2 = k.rr2;
    float* ysl = k.YS + (w * PBY + k.hf * RPL) * W + xo;   // plane w - 1 (YS holds planes -1..BZ)
    const float* hs = k.HS + C * NH * W + xo;
    const bool act = !RAG || k.act;
    const int top = RAG ? k.planes : BZ;   // planes of the brick
    const int s = C ? N - j : j + 1;
    const int sp = s <= k.nA ? 0 : 1;
    const bool acc = C ? j >= N - hm : j >= hm;
    if (j > 0) bar_wait(k.full + C, (unsigned)((j - 1) & 1), k.ctl, k.dead);
    // the rows next to the lane's first and last row: y-halo rows, or across the lane halves
    float up[VEC], dn[VEC];
    if constexpr (RG::HALVES == 2) {
        float v[VEC], o[VEC];
        ldv<VEC>(hs + halo_row<PBY, BZ>(k.hf ? PBY : -1, w) * W, v);
        xpassv<VEC>(k, v, o);
#pragma unroll
        for (int i = 0; i < VEC; ++i) {
            const float last = __shfl_xor_sync(0xffffffffu, xf[RPL - 1][i], LPR);
            const float first = __shfl_xor_sync(0xffffffffu, xf[0][i], LPR);
            up[i] = k.hf ? last : o[i];
            dn[i] = k.hf ? o[i] : first;
        }
    } else {
        float v[VEC], u[VEC];
        ldv<VEC>(hs + halo_row<PBY, BZ>(-1, w) * W, v);
        ldv<VEC>(hs + halo_row<PBY, BZ>(PBY, w) * W, u);
        xpassv<VEC>(k, v, up);
        xpassv<VEC>(k, u, dn);
    }
    // every warp has read YS of the previous unit
    if (C) bar_wait(k.pub, (unsigned)(j & 1), k.ctl, k.dead);
    else if (j > 0) bar_wait(k.pub + 1, (unsigned)((j - 1) & 1), k.ctl, k.dead);
    // z-halo planes, one row per lane half: y pass of the raw rows, then the x pass
#pragma unroll
    for (int t0 = w * RG::HALVES; t0 < 2 * PBY; t0 += NW * RG::HALVES) {
        const int t = t0 + k.hf;
        const int side = t / PBY, r = t % PBY, pl = side ? BZ : -1;
        float a[VEC], c[VEC], d[VEC], m[VEC], o[VEC];
        ldv<VEC>(hs + halo_row<PBY, BZ>(r - 1, pl) * W, a);
        ldv<VEC>(hs + halo_row<PBY, BZ>(r, pl) * W, c);
        ldv<VEC>(hs + halo_row<PBY, BZ>(r + 1, pl) * W, d);
        mixv<VEC>(a, c, d, rr, rr2, m);
        xpassv<VEC>(k, m, o);
        stv<VEC>(k.YS + ((side ? top + 1 : 0) * PBY + r) * W + xo, o);
    }
    {
        float* yw = ysl + PBY * W;
        float prev[VEC];
#pragma unroll
        for (int i = 0; i < VEC; ++i) prev[i] = up[i];
#pragma unroll
        for (int p = 0; p < RPL; ++p) {
            float yv[VEC], cur[VEC];
#pragma unroll
            for (int i = 0; i < VEC; ++i) cur[i] = xf[p][i];
            if (p + 1 < RPL) mixv<VEC>(prev, cur, xf[p + 1 < RPL ? p + 1 : p], rr, rr2, yv);
            else mixv<VEC>(prev, cur, dn, rr, rr2, yv);
#pragma unroll
            for (int i = 0; i < VEC; ++i) {
                prev[i] = cur[i];
                xf[p][i] = yv[i];   // xf now holds the y-filtered rows
            }
            if (act) stv<VEC>(yw + p * W, yv);   // (an idle warp's place may be the upper halo plane's)
        }
    }
    compute_sync(32 * NW);
    if (acc) cp_wait_all();   // the thread's own stack values of this unit
    // z pass and step output.  The boundary rows go first and are published; the interior of a stored
    // level (no interior is stored past the middle) follows with the x pass.
    const bool last = j + 1 == N;
    float* dst = level_of(k.A, C, N, hm, j) + k.own;
    const unsigned te = k.tbase + (unsigned)(sp * 32), ta = te + 64u;
    const int hf = k.hf;
    auto edge_row = [&](int p) { return k.face_plane || (p == 0 && hf == 0) || (p == RPL - 1 && hf == RG::HALVES - 1); };
    float e2[2][VS], q2[2][VS];   // Boltzmann factors and quadrature of this row and the next
#pragma unroll
    for (int i = 0; i < VS; ++i) q2[0][i] = q2[1][i] = 0.f;
    tm_ld<VS>(te, e2[0]);
    if (acc) tm_ld<VS>(ta, q2[0]);
#pragma unroll
    for (int p = 0; p < RPL; ++p) {
        tm_wait_ld<VS>(e2[p & 1], q2[p & 1]);
        if (p + 1 < RPL) {
            tm_ld<VS>(te + (p + 1) * VS, e2[(p + 1) & 1]);
            if (acc) tm_ld<VS>(ta + (p + 1) * VS, q2[(p + 1) & 1]);
        }
        float a[VEC], d[VEC], sg[VEC], e[VEC], out[VEC];
        ldv<VEC>(ysl + p * W, a);
        ldv<VEC>(ysl + (2 * PBY + p) * W, d);
        mixv<VEC>(a, xf[p], d, rr, rr2, sg);
#pragma unroll
        for (int i = 0; i < VEC; ++i) e[i] = e2[p & 1][i];
        mulv<VEC>(e, sg, out);
        if (acc) {   // q_I += sigma[own chain] x (the other chain's stored value)
            float st[VEC], q[VEC];
            ldv<VEC>(k.GS + p * W, st);
#pragma unroll
            for (int i = 0; i < VEC; ++i) q[i] = q2[p & 1][i];
            fmav<VEC>(st, sg, q);
#pragma unroll
            for (int i = 0; i < VEC; ++i) q2[p & 1][i] = q[i];
            tm_st<VS>(ta + p * VS, q2[p & 1]);
        }
        if (edge_row(p) && !last && act) stg<VEC>(dst + p * W, out);
        if (C == 0 && last && act) {
            float t = out[0] + out[1];
            if constexpr (VEC == 3) t = t + out[2];
            if constexpr (VEC == 4) t = t + (out[2] + out[3]);
            k.qsum += t;
        }
#pragma unroll
        for (int i = 0; i < VEC; ++i) xf[p][i] = out[i];
    }
    if (acc) tm_wait_st();
    __syncwarp();
    if (k.lane == 0) bar_arrive(k.pub + C);
    if (!acc) {
#pragma unroll
        for (int p = 0; p < RPL; ++p)
            if (!edge_row(p) && act) stg<VEC>(dst + p * W, xf[p]);
    }
    // The next unit's stack level (the other chain's), if that unit accumulates: every thread copies
    // the values of its own sites, which it stored itself, and brings the line that the chain after
    // it takes next into L2 meanwhile.
    {
        const int jn = C ? j + 1 : j;
        if ((C ? jn >= hm : jn >= N - hm) && jn < N && act) {
            const float* src = k.A.stack + (size_t)(C ? jn : N - jn - 1) * k.A.V;
#pragma unroll
            for (int p = 0; p < RPL; ++p) cpv<VEC>(k.GS + p * W, src + k.own + p * W);
            if (k.lane * 32 < PBY * W && jn + 1 < N)
                asm volatile("prefetch.global.L2 [%0];\n" ::"l"(C ? src + k.A.V + k.slab : src - k.A.V + k.slab));
        }
    }
#pragma unroll
    for (int p = 0; p < RPL; ++p) {
        float o[VEC];
        xpassv<VEC>(k, xf[p], o);
#pragma unroll
        for (int i = 0; i < VEC; ++i) xf[p][i] = o[i];
    }
}

}  // namespace

size_t pers_smem_bytes(int width, int pby, int bz) {
    const size_t PBY = (size_t)pby;
    // YS (y-filtered level, planes -1..bz) + raw halo rows of both chains + stack values
    const size_t rows = (size_t)(bz + 2) * PBY + 2 * 2 * (bz + 2 + PBY) + (size_t)bz * PBY;
    return rows * (size_t)width * sizeof(float);
}

// Warp w < NW owns plane w of the brick, all PBY rows (HALVES rows side by side), VEC sites of each
// row per lane, of both chains.  What bounds a unit (clock64 per phase, 128 x 8 x 16 bricks, about
// 6000 cycles): the shared-memory pipe (y-filtered rows written once and read twice, halo and stack
// rows, shuffles: about 2500 cycles of it before the middle and 3700 past it) and the latencies
// between the barriers.
//
// RAG: the planes need not be a multiple of BZ; the uppermost bricks then have the remainder (a multiple of
// 8), and the warps beyond it only take part in the halo planes and the barriers.  For grids with more
// bricks of 8 planes than SMs, two of which do not fit one (the tensor memory).  Density evaluations, N = 48,
// two bricks per SM (the kernels before these), the general sweeps, and so: 128 x 128 x 136 527, 573 and 342 us;
// 64 x 256 x 136 520, 691, 359; 32 x 256 x 120 407, 572, 239; 96 x 128 x 120 475, 486, 367.
template <int W, int PBY, int BZ, int NW, bool RAG>
__device__ __forceinline__ void pers_sweep(const Rep* __restrict__ reps, const PersCtl& ctl) {
    static_assert(NW == BZ, "one warp per plane");
    using RG = PRow<W, PBY>;
    constexpr int VEC = RG::VEC, LPR = RG::LPR, RPL = RG::RPL;
    constexpr int VS = VEC == 3 ? 4 : VEC;   // tensor-memory columns of a row's sites
    constexpr int NH = 2 * (BZ + 2 + PBY), CH = W / 4;   // halo rows; 16-byte chunks per row
    constexpr int TCOLS = 128 * (NW / 4);    // 4 regions of 32 columns per warp, 4 warps side by side
    static_assert(RPL * VS <= 32, "tensor-memory columns");
    extern __shared__ __align__(128) unsigned char smem[];
    float* YS = (float*)smem;                                  // [BZ+2][PBY][W]
    float* HS = YS + (BZ + 2) * PBY * W;                       // [2][NH][W] raw halo rows of each chain
    float* GS = HS + 2 * NH * W;                               // [BZ][PBY][W] stack values
    __shared__ double sh[33];
    __shared__ int nbs[8];
    __shared__ PersArrays arr;
    __shared__ __align__(8) unsigned long long full[2], pub[2];
    __shared__ unsigned tmem_slot;
    const int4 tb = ctl.table[blockIdx.x];
    const Rep& R = reps[tb.x];
    const int b = tb.y;
    const int ny = R.ny, nz = R.nz, N = R.N, nA = R.nA;
    const int plane = W * ny;
    const size_t V = (size_t)R.V;
    const int nby = ny / PBY, nbz = RAG ? (nz + BZ - 1) / BZ : nz / BZ;
    const int by = b % nby, bz = b / nby;
    const int y0 = by * PBY, z0 = bz * BZ;
    const int planes = RAG ? min(BZ, nz - z0) : BZ;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    int* fown = ctl.flags + (size_t)(tb.z + tb.y) * kFlagStride;   // own step counters: +0 forward, +kFlagChain
    if (threadIdx.x < 8) {
        const int k = threadIdx.x < 4 ? threadIdx.x : threadIdx.x + 1;   // skip the centre
        const int dy = k % 3 - 1, dz = k / 3 - 1;
        nbs[threadIdx.x] = tb.z + (by + dy + nby) % nby + nby * ((bz + dz + nbz) % nbz);
    }
    if (threadIdx.x < 4)
        arr.exch[threadIdx.x >> 1][threadIdx.x & 1] =
            (float*)(threadIdx.x == 0 ? R.del0 : threadIdx.x == 1 ? R.del1 : threadIdx.x == 2 ? R.Gp0 : R.Gp1);
    if (threadIdx.x == 4) arr.stack = (float*)R.G;
    if (threadIdx.x == 5) arr.V = V;
    // the first inputs: G_0 = 1 and G+_{N+1} = 1
    for (int i = threadIdx.x; i < 2 * NH * W; i += 32 * (NW + kXWarps)) HS[i] = 1.0f;
    if (w == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(saddr(&tmem_slot)), "r"(TCOLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
    }
    if (threadIdx.x == 0) {
        for (int c = 0; c < 2; ++c) {
            bar_init(&full[c], 64);
            bar_init(&pub[c], NW);
        }
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    // step counters of a replica's bricks are equal at launch (unsigned: they may wrap in long runs);
    // read by both of a chain's exchange warps before either publishes
    const unsigned c0 = w >= NW ? (unsigned)fown[((w - NW) >> 1) * kFlagChain] : 0u;
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");

    if (w >= NW) {
        // ---- exchange warps, two per chain: per step publish, wait for the neighbours, copy halo rows ----
        regs_dec<PersRegs<NW>::exchange>();
        const int c = (w - NW) >> 1, part = (w - NW) & 1;   // part 0: rows -1 and plane -1, 1: rows PBY and plane BZ
        fown += c * kFlagChain;
        bool aborted = ld_acquire(ctl.abort) != 0, dead = false;
        const int* nbf = ctl.flags + (size_t)nbs[lane & 7] * kFlagStride + c * kFlagChain;
        constexpr int RPI = 32 / CH;                        // rows a warp copies at once
        const int lr = lane / CH, lc = 4 * (lane - lr * CH);
        float* hdst = HS + (c * NH + part * (NH / 2) + lr) * W + lc;
        const int yrow = (part ? (y0 + PBY == ny ? 0 : y0 + PBY) : (y0 == 0 ? ny - 1 : y0 - 1)) * W + lc;
        const int zpl = (part ? (z0 + planes == nz ? 0 : z0 + planes) : (z0 == 0 ? nz - 1 : z0 - 1)) * plane + y0 * W + lc;
        for (int j = 0; j < N; ++j) {
            bar_wait(&pub[c], (unsigned)(j & 1), ctl, dead);
            // pub orders every warp's boundary stores before this release store, and release is
            // cumulative, so a CTA whose acquire load reads the new counter sees them
            const unsigned target = c0 + (unsigned)j + 1u;
            if (part == 0 && lane == 0) st_release(fown, (int)target);
            if (j + 1 >= N) break;
            // lanes 0..7 poll one neighbour each; every 32 polls they look at the abort flag
            if (lane < 8 && !aborted) {
                int spins = 0;
                while ((int)((unsigned)ld_acquire(nbf) - target) < 0) {   // wrap-safe: counters only grow
                    if ((++spins & 31) == 0) {
                        if (ld_acquire(ctl.abort) != 0) {
                            aborted = true;
                            break;
                        }
                        if (spins > ctl.limit) {
                            atomicOr(ctl.status, (int)ST_TIMEOUT);
                            atomicExch(ctl.abort, 1);
                            aborted = true;
                            break;
                        }
                    }
                    __nanosleep(32);
                }
            }
            aborted = __any_sync(0xffffffffu, aborted);
            const float* src = level_of(arr, c, N, (N + 1) / 2, j);
            if (lr < RPI) {
#pragma unroll 3
                for (int i0 = 0; i0 < BZ + 2; i0 += RPI) {   // row -1 (PBY) of planes -1..BZ
                    const int i = i0 + lr;                  // (slot BZ + 1: the plane above the brick)
                    int z = RAG && i == BZ + 1 ? z0 + planes : z0 - 1 + i;
                    z = z < 0 ? z + nz : (z >= nz ? z - nz : z);
                    if (RAG && i > planes && i <= BZ) continue;
                    if ((BZ + 2) % RPI == 0 || i < BZ + 2) cp16(hdst + i0 * W, src + z * plane + yrow);
                }
#pragma unroll 2
                for (int i0 = 0; i0 < PBY; i0 += RPI)        // the own rows of plane -1 (BZ)
                    cp16(hdst + (BZ + 2 + i0) * W, src + zpl + (i0 + lr) * W);
            }
            cp_arrive(&full[c]);
        }
    } else {
        // ---- compute warps ----
        regs_inc<PersRegs<NW>::compute>();
        const int hf = lane / LPR, li = lane - hf * LPR;   // lane half (row group) and lane within the row
        const int xo = VEC * li;
        const int seg = lane - li;
        const int lsrc = seg + ((li + LPR - 1) & (LPR - 1)), rsrc = seg + ((li + 1) & (LPR - 1));
        // Each 1-D pass is applied as c + r (a + d) with r = alpha / (1 - 2 alpha), i.e. the
        // stencil's pass divided by its centre weight; the Boltzmann factors carry a weight against the
        // growth (Par::ew), and the normalisation takes both into account.
        const float rr = R.pf.rr;
        // own plane never wraps: (row r, plane w) is own0 + r * W
        const size_t own0 = (size_t)(z0 + w) * plane + (size_t)(y0 + hf * RPL) * W + xo;
        PersWarp k = {arr, ctl, full, pub, YS, HS, GS + (w * PBY + hf * RPL) * W + xo, own0,
                      (size_t)(z0 + w) * plane + (size_t)y0 * W + 32 * lane,
                      N, nA, (N + 1) / 2, w, lane, hf, xo, lsrc, rsrc, planes, w < planes, w == 0 || w == planes - 1, rr, pk2(rr, rr),
                      tmem_slot + ((unsigned)((w & 3) * 32) << 16) + (unsigned)((w >> 2) * 128), 0.f, false};
        const unsigned tbase = k.tbase;

        // tensor memory regions: 0, 1 Boltzmann factors of A, B; 2, 3 quadratures
#pragma unroll
        for (int I = 0; I < 2; ++I) {
            const float* E = (const float*)R.E + (size_t)I * V;
#pragma unroll
            for (int p = 0; p < RPL; ++p) {
                float t[VS], zero[VS], e[VEC] = {};
                if (!RAG || k.act) ldv<VEC>(E + own0 + (size_t)p * W, e);
#pragma unroll
                for (int i = 0; i < VS; ++i) {
                    t[i] = i < VEC ? e[i < VEC ? i : 0] : 0.f;
                    zero[i] = 0.f;
                }
                tm_st<VS>(tbase + I * 32 + p * VS, t);
                tm_st<VS>(tbase + (2 + I) * 32 + p * VS, zero);
            }
        }
        tm_wait_st();

        const float one = 1.0f + 2.0f * rr;   // the x pass of G_0 = 1 and of G+_{N+1} = 1
        float xF[RPL][VEC], xB[RPL][VEC];
#pragma unroll
        for (int p = 0; p < RPL; ++p)
#pragma unroll
            for (int i = 0; i < VEC; ++i) xF[p][i] = xB[p][i] = one;

#pragma unroll 1
        for (int j = 0; j < N; ++j) {
            pers_unit<W, PBY, BZ, NW, RAG, 0>(k, xF, j);
            pers_unit<W, PBY, BZ, NW, RAG, 1>(k, xB, j);
        }
        // both quadratures
#pragma unroll
        for (int I = 0; I < 2; ++I) {
            float* q = (float*)R.q + (size_t)I * V;
#pragma unroll
            for (int p = 0; p < RPL; ++p) {
                float t[VS], o[VEC];
                tm_ld<VS>(tbase + (2 + I) * 32 + p * VS, t);
                tm_wait_ld<VS>(t);
#pragma unroll
                for (int i = 0; i < VEC; ++i) o[i] = t[i];
                if (!RAG || k.act) stv<VEC>(q + own0 + (size_t)p * W, o);
            }
        }
        // the brick's share of Q, the end of the tensor memory's use (compute warps only: the
        // exchange warps hold too few registers to join code that follows both branches)
        const double t = warp_sum((double)k.qsum);
        if (lane == 0) sh[w] = t;
        asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
        compute_sync(32 * NW);
        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
        if (w == 0) {
            const double q = warp_sum(lane < NW ? sh[lane] : 0.0);
            // the replica's last brick adds up all bricks' shares, in order
            const int nb = nby * nbz;
            unsigned old = 0;
            if (lane == 0) {
                slot(R, P_Q)[b] = q;
                __threadfence();
                old = atomicInc((unsigned*)(R.scal + S_QFIN), (unsigned)nb - 1u);
            }
            if (__shfl_sync(0xffffffffu, old, 0) == (unsigned)nb - 1u) {
                __threadfence();
                double s = 0.0;
                for (int i = lane; i < nb; i += 32) s += __ldcg(slot(R, P_Q) + i);
                s = warp_sum(s);
                if (lane == 0) R.scal[S_QSUM] = s;
            }
            asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem_slot), "r"(TCOLS) : "memory");
        }
    }
}

template <int W, int PBY, int BZ, int NW, bool RAG = false>
__global__ void __launch_bounds__(32 * (NW + kXWarps), 1) k_prop_pers(const Rep* __restrict__ reps, PersCtl ctl) {
    pers_sweep<W, PBY, BZ, NW, RAG>(reps, ctl);
}

// Bricks of several row widths (32 to 96 sites) in one launch (batches): each CTA runs the sweep of
// its replica's width; the launch's dynamic shared memory covers the largest.  128-wide replicas
// keep launches of their own (with them in the same function the registers would spill).
template <int BZ, int NW>
__global__ void __launch_bounds__(32 * (NW + kXWarps), 1) k_prop_pers_mix(const Rep* __restrict__ reps, PersCtl ctl) {
    const Rep& R = reps[ctl.table[blockIdx.x].x];
    const int pby = pers_pby_of(R.nx, R.ny);
    switch (R.nx * 32 + pby) {
        case 32 * 32 + 8: pers_sweep<32, 8, BZ, NW, false>(reps, ctl); break;
        case 32 * 32 + 16: pers_sweep<32, 16, BZ, NW, false>(reps, ctl); break;
        case 48 * 32 + 8: pers_sweep<48, 8, BZ, NW, false>(reps, ctl); break;
        case 48 * 32 + 16: pers_sweep<48, 16, BZ, NW, false>(reps, ctl); break;
        case 64 * 32 + 8: pers_sweep<64, 8, BZ, NW, false>(reps, ctl); break;
        case 64 * 32 + 16: pers_sweep<64, 16, BZ, NW, false>(reps, ctl); break;
        case 96 * 32 + 8: pers_sweep<96, 8, BZ, NW, false>(reps, ctl); break;
        default: break;   // not reached: the host builds mixed launches of these widths only
    }
}

// Host side ---------------------------------------------------------------------------------

bool pers_width_ok(int nx) { return nx == 32 || nx == 48 || nx == 64 || nx == 96 || nx == 128; }

int pers_pby(const Rep& R) { return pers_pby_of(R.nx, R.ny); }

size_t pers_mix_smem_bytes(int bz) {
    size_t m = 0;
    for (int w : {32, 48, 64}) m = std::max(m, pers_smem_bytes(w, 16, bz));
    for (int w : {32, 48, 64, 96}) m = std::max(m, pers_smem_bytes(w, 8, bz));
    return m;
}

// Brick depths: 16 planes on 16 warps or 8 planes on 8 warps.  (Grids of up to two shallow bricks per SM
// are accepted; more than one do not run together, and such grids take bricks of 16 planes, the uppermost
// of 8 where 16 does not divide nz, or the general sweeps.)
bool pers_supported(const Rep& R, int bz, int nw, int nsm) {
    if (!pers_width_ok(R.nx) || R.ny % 8 || R.nz % bz) return false;
    if (!((bz == 16 && nw == 16) || (bz == 8 && nw == 8))) return false;   // one warp per plane
    const int nb = pers_bricks(R, bz);
    return nb >= 1 && nb <= nsm * (nw == 8 ? 2 : 1);   // all bricks co-resident
}

int pers_bricks(const Rep& R, int bz) { return (R.ny / pers_pby(R)) * ((R.nz + bz - 1) / bz); }

namespace {
// Also checks that the registers the kernel launches with cover the shares its warps take
// (setmaxnreg would wait for ever if they did not).
template <int NW, typename K>
cudaError_t pers_attr_of(K kernel, size_t smem) {
    cudaFuncAttributes fa;
    cudaError_t e = cudaFuncGetAttributes(&fa, kernel);
    if (e == cudaSuccess &&
        fa.numRegs * (NW + kXWarps) < PersRegs<NW>::compute * NW + PersRegs<NW>::exchange * kXWarps)
        e = cudaErrorInvalidConfiguration;
    if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
    return e;
}
template <int W, int PBY, int BZ, int NW, bool RAG = false>
cudaError_t pers_attr() {
    return pers_attr_of<NW>(k_prop_pers<W, PBY, BZ, NW, RAG>, pers_smem_bytes(W, PBY, BZ));
}
template <int BZ, int NW>
cudaError_t pers_mix_attr() {
    return pers_attr_of<NW>(k_prop_pers_mix<BZ, NW>, pers_mix_smem_bytes(BZ));
}
}  // namespace

// ACTION(W, PBY, BZ, NW) for the instantiated (width, rows) pairs of one brick depth
#define DSCF_PERS_SWITCH(BB, NN, ACTION)                          \
    switch (width * 32 + pby) {                                  \
        case 128 * 32 + 8: ACTION(128, 8, BB, NN); break;        \
        case 96 * 32 + 8: ACTION(96, 8, BB, NN); break;          \
        case 64 * 32 + 8: ACTION(64, 8, BB, NN); break;          \
        case 64 * 32 + 16: ACTION(64, 16, BB, NN); break;        \
        case 48 * 32 + 8: ACTION(48, 8, BB, NN); break;          \
        case 48 * 32 + 16: ACTION(48, 16, BB, NN); break;        \
        case 32 * 32 + 8: ACTION(32, 8, BB, NN); break;          \
        case 32 * 32 + 16: ACTION(32, 16, BB, NN); break;        \
        default: break;                                          \
    }

int pers_prepare(int width, int pby, int bz, int nw, bool rag) {
    cudaError_t e = cudaErrorInvalidValue;
#define DSCF_PERS_ATTR(WW, PP, BB, NN) e = pers_attr<WW, PP, BB, NN>()
#define DSCF_PERS_ATTR_RAG(WW, PP, BB, NN) e = pers_attr<WW, PP, BB, NN, true>()
    if (rag) {
        DSCF_PERS_SWITCH(16, 16, DSCF_PERS_ATTR_RAG)
    } else if (bz == 16 && nw == 16) {
        if (width == 0) e = pers_mix_attr<16, 16>();
        else DSCF_PERS_SWITCH(16, 16, DSCF_PERS_ATTR)
    } else if (bz == 8 && nw == 8) {
        if (width == 0) e = pers_mix_attr<8, 8>();
        else DSCF_PERS_SWITCH(8, 8, DSCF_PERS_ATTR)
    }
#undef DSCF_PERS_ATTR
#undef DSCF_PERS_ATTR_RAG
    return (int)e;
}

namespace {
// The SM that runs each CTA of a launch shaped like the sweep (same block size, shared memory
// and cooperative attribute), for the placement of bricks on SMs.
template <int NW>
__global__ void __launch_bounds__(32 * (NW + kXWarps), 1) k_pers_place(int* smid) {
    if (threadIdx.x == 0) {
        unsigned id;
        asm volatile("mov.u32 %0, %%smid;" : "=r"(id));
        smid[blockIdx.x] = (int)id;
    }
}
}  // namespace

int pers_placement(int bz, int nw, int nbricks, int* d_smid, cudaStream_t stream) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(nbricks);
    cfg.blockDim = dim3(32 * (nw + kXWarps));
    cfg.dynamicSmemBytes = pers_smem_bytes(128, 8, bz);
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cudaError_t e;
    if (nw == 16) {
        e = cudaFuncSetAttribute(k_pers_place<16>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)cfg.dynamicSmemBytes);
        if (e == cudaSuccess) e = cudaLaunchKernelEx(&cfg, k_pers_place<16>, d_smid);
    } else {
        e = cudaFuncSetAttribute(k_pers_place<8>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)cfg.dynamicSmemBytes);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(k_pers_place<8>, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
        if (e == cudaSuccess) e = cudaLaunchKernelEx(&cfg, k_pers_place<8>, d_smid);
    }
    return (int)e;
}

int launch_prop_pers(const Launch& L, int width, int pby, int bz, int nw, bool rag, int nbricks, const int4* table,
                     int* flags, int* abortf, int limit) {
    PersCtl ctl;
    ctl.flags = flags;
    ctl.abort = abortf;
    ctl.status = L.status;
    ctl.table = table;
    ctl.limit = limit;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(nbricks);
    cfg.blockDim = dim3(32 * (nw + kXWarps));
    cfg.dynamicSmemBytes = width ? pers_smem_bytes(width, pby, bz) : pers_mix_smem_bytes(bz);
    cfg.stream = L.stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cudaError_t e = cudaErrorInvalidValue;
#define DSCF_PERS_LAUNCH(WW, PP, BB, NN) e = cudaLaunchKernelEx(&cfg, k_prop_pers<WW, PP, BB, NN>, L.reps, ctl)
#define DSCF_PERS_LAUNCH_RAG(WW, PP, BB, NN) e = cudaLaunchKernelEx(&cfg, k_prop_pers<WW, PP, BB, NN, true>, L.reps, ctl)
    if (rag) {
        DSCF_PERS_SWITCH(16, 16, DSCF_PERS_LAUNCH_RAG)
    } else if (bz == 16 && nw == 16) {
        if (width == 0) e = cudaLaunchKernelEx(&cfg, k_prop_pers_mix<16, 16>, L.reps, ctl);
        else DSCF_PERS_SWITCH(16, 16, DSCF_PERS_LAUNCH)
    } else if (bz == 8 && nw == 8) {
        if (width == 0) e = cudaLaunchKernelEx(&cfg, k_prop_pers_mix<8, 8>, L.reps, ctl);
        else DSCF_PERS_SWITCH(8, 8, DSCF_PERS_LAUNCH)
    }
#undef DSCF_PERS_LAUNCH
#undef DSCF_PERS_LAUNCH_RAG
    return (int)e;
}
#undef DSCF_PERS_SWITCH

}  // namespace dscf
