// General contour sweeps (Eq. 16-17): any grid, both precisions, one replica or a batch of unlike
// ones, in one launch.
//
// A cooperative launch of one CTA per SM runs both chains of a density evaluation level by level.
// Like the brick kernel's (dscf_pers.cu), the forward chain G_s and the backward one G+_s meet in the
// middle, h = ceil(N / 2): each stores its levels up to there in the contour stack (G_s, s <= h;
// G+_s, s > h) and past it multiplies sigma of its own field with the stored value of the other,
// q_{I_s} += sigma[G_{s-1}] G+_s = G_s sigma[G+_{s+1}].  A chain's level needs the whole previous
// level, so a counter per chain is the grid's barrier between levels; a CTA arrives at one chain's
// barrier, computes its share of the other chain's level and only then waits, so that the barrier's
// L2 round trips overlap with work (a warp per chain arrives and polls; the compute warps only meet
// it in shared memory).
//
// Work is cut into runs of consecutive z planes of one x row (or one x tile of a row of more than 256
// sites), spread over all warps of the launch (coop_cut).  A warp marches its run: per plane it loads the
// row and its two y neighbours, applies the y pass, then the x pass by shuffles (lane L holds sites L,
// L + 32, ... of the row, so any row length and alignment has coalesced accesses), and combines three
// planes in registers.  No pass is computed twice but the y and x passes of the two planes beside a
// run, no shared memory and no barrier inside a level, and each pass is one add and one fma
// (c + r (a + d), r = alpha / (1 - 2 alpha), the centre weights made up for by the Boltzmann factors and the
// normalisation): 7 operations a site and contour step forward, 8 with the quadrature.
//
// FP64 at 128^3 is bound by the FP64 pipe (31 us of operations in a level's 33 us), 256^3 by HBM (592 MB
// a pair of levels at 77% of the copy rate), the rest by the latency of loads and of the barrier: hence loads
// several planes ahead, 12 warps where the registers allow it (128^3 FP32: 750 us with 8, 689 with 12) and one run per warp.
// A density evaluation, one launch per contour step and direction, and so: 32^3, N = 32, FP64 539 -> 126 us;
// 100 x 90 x 75, N = 48, FP32 1013 -> 274 us; 128^3, N = 64, FP64 8.9 -> 4.2 ms; 256^3, N = 64, FP32 8.07
// (fused pairs of steps) -> 7.25 ms.  Against the brick sweeps (dscf_pers.cu): 48^3, N = 16 71 us (bricks 137),
// 64^3, N = 64 241 (361), 96^3, N = 48 347 (227), 128^3, N = 64 689 (386).
//
// Every wait is bounded as in dscf_pers.cu: a CTA that runs out sets the status bit and the abort flag
// and waits no more; arrivals do not depend on waits, so the launch always finishes and leaves its
// counters at zero.
// Included by dscf_coop32.cu and dscf_coop64.cu, one per precision, and by dscf_coop32m.cu and dscf_coop64m.cu
// for the kernels that hold every row layout (they compile in parallel).
#pragma once
#include "dscf_internal.cuh"

#include <cstring>

// the row layouts that coop_layout() gives: (sites per lane, mode)
#define DSCF_COOP_LAYOUTS(X)                                                                                \
    X(1, BLOCKED) X(2, BLOCKED) X(3, BLOCKED) X(4, BLOCKED) X(6, BLOCKED) X(8, BLOCKED) X(2, STRIDED) \
    X(3, STRIDED) X(4, STRIDED) X(5, STRIDED) X(6, STRIDED) X(7, STRIDED) X(8, STRIDED) X(4, TILE) X(5, TILE) \
    X(4, BTILE)
#define DSCF_COOP_LAYOUTS32(X) X(2, ROWS) X(4, ROWS)   // in FP32 only

namespace dscf {

namespace {

struct CoopCtl {
    const CoopRep* reps;         // replicas by decreasing chain length
    int nrep;
    int j0, j1;                  // levels of this launch
    int* cnt;                    // barrier counters: chain c at c * kFlagStride, exits at 2 * kFlagStride
    int* abort;
    int* status;
    int limit;                   // polls before giving up
    int runs, per;               // runs > 0: one replica, one run of a row per warp, `per` warps of a CTA
};

__device__ __forceinline__ void red_release(int* p) {
    asm volatile("red.release.gpu.global.add.s32 [%0], 1;\n" ::"l"(p) : "memory");
}

// One chain's level on one replica.
template <typename T>
struct CoopOps {
    const T* src;   // previous level; nullptr: the constant field 1
    T* dst;         // nullptr: the level is not needed
    const T* E;
    const T* st;    // stored level of the other chain (quadrature), nullptr before the middle
    T* q;           // quadrature
    bool first;     // q starts here
    bool lastQ;     // sum the level (G_N)
    double* qrow;   // its sums per row plane, or nullptr: one sum per warp
};

// Level i of chain C (contour step s = i + 1 forward, s = N - i backward).  Before the chains meet it is
// stored at its bead's place in the stack.  Past the middle a chain overwrites the place of its bead,
// whose value of the other chain it has just used at the same site (and thread), except at its
// first level there: that place is still the other chain's input, so the level goes to a field of its
// own.  (A later place was last read as a neighbour at least one full level of both chains earlier.)
template <typename T, int C>
__device__ __forceinline__ CoopOps<T> coop_ops(const CoopRep& R, int j) {
    CoopOps<T> o;
    const size_t V = (size_t)R.V;
    const int N = R.N, nA = R.nA, h = (N + 1) / 2;
    const int s = C ? N - j : j + 1, sp = s <= nA ? 0 : 1;
    T* stack = (T*)R.G;
    const int mid = C ? N - h : h;
    auto level = [&](int i) -> T* {
        if (i == mid) return (T*)(C ? R.Gp1 : R.Gp0);
        return stack + (size_t)(C ? N - i - 1 : i) * V;
    };
    o.src = j == 0 ? nullptr : level(j - 1);
    o.dst = j == N - 1 ? nullptr : level(j);   // the last level of a chain is not read again (Q is summed in registers)
    o.E = (const T*)R.E + (sp ? V : 0);
    o.st = j >= mid ? stack + (size_t)(s - 1) * V : nullptr;
    o.q = (T*)R.q + (sp ? V : 0);
    // A block's quadrature starts at its first bead past the middle on either side.  Where beads of
    // one block lie on both sides both chains add to it: the same thread, in the order of the units
    // (backward first for odd N).
    const bool both = nA != h;   // the block of beads h and h + 1
    o.first = C ? ((j == mid && !(both && (N & 1) == 0)) || s == nA) : ((j == mid && !(both && (N & 1))) || s == nA + 1);
    o.lastQ = !C && j == N - 1;
    o.qrow = R.qrow;
    return o;
}

// Layout of a row over a warp's lanes, from its length (coop_layout):
//   blocked: lane L holds sites K L .. K L + K - 1 (K divides nx, nx / K <= 32 lanes): vector
//            accesses, two shuffles for the x pass;
//   strided: lane L holds sites L, L + 32, ... (any nx <= 256): scalar accesses, 2 K + 2 shuffles;
//   tile:    like strided, of columns x0 - 1 .. x0 + tile of which the outer two are neighbours (nx > 256);
//   btile:   like blocked, the first and the last lane hold the neighbours' sites (nx > 256, 4 | nx);
//   rows:    blocked, several adjacent rows side by side (even nx <= 32 in FP32 fields of many rows).
// Rows of more than 256 sites, density evaluations of N = 24, us, by the kernels before these (a launch per
// level), in whole strided tiles of 254 columns (300 columns then cost 512), and in equal tiles:
//   512 x 128 x 128 FP32 2570, 4713, 1794, FP64 11608, 14301, 7656;  300 x 300 x 100 FP32 2650, 5330, 1921;
//   1024 x 64 x 64 FP32 1408, 2652, 795;  257 x 40 x 40 FP32 446, 510, 216, FP64 1064, 1156, 652.
enum { BLOCKED = 0, STRIDED = 1, TILE = 2, BTILE = 3, ROWS = 4 };

// K values of a lane at p: one access of 16, 8 or 4 bytes each where their size allows.
template <typename T, int K>
__device__ __forceinline__ void ldk(const T* p, T (&v)[K]) {
    constexpr int B = K * (int)sizeof(T);
    if constexpr (B % 16 == 0) {
#pragma unroll
        for (int i = 0; i < B / 16; ++i) {
            const int4 t = ((const int4*)p)[i];
            memcpy((char*)&v[0] + 16 * i, &t, 16);
        }
    } else if constexpr (B % 8 == 0 && sizeof(T) == 4) {
#pragma unroll
        for (int i = 0; i < B / 8; ++i) {
            const float2 t = ((const float2*)p)[i];
            v[2 * i] = t.x;
            v[2 * i + 1] = t.y;
        }
    } else {
#pragma unroll
        for (int i = 0; i < K; ++i) v[i] = p[i];
    }
}
template <typename T, int K>
__device__ __forceinline__ void stk(T* p, const T (&v)[K]) {
    constexpr int B = K * (int)sizeof(T);
    if constexpr (B % 16 == 0) {
#pragma unroll
        for (int i = 0; i < B / 16; ++i) {
            int4 t;
            memcpy(&t, (const char*)&v[0] + 16 * i, 16);
            ((int4*)p)[i] = t;
        }
    } else if constexpr (B % 8 == 0 && sizeof(T) == 4) {
#pragma unroll
        for (int i = 0; i < B / 8; ++i) ((float2*)p)[i] = make_float2(v[2 * i], v[2 * i + 1]);
    } else {
#pragma unroll
        for (int i = 0; i < K; ++i) p[i] = v[i];
    }
}

// n planes from za of x row (or x tile at x0) y.  PAST: past the middle (stored levels of the other chain are
// read and the quadrature grows).  The march is bound by the latency of its loads, so those of a plane are
// issued D planes (rows) and two planes (operands of the output plane) ahead; rings are registers by name, the
// loop is unrolled by their length.
template <typename T, int K, int MODE, bool PAST>
__device__ __forceinline__ void coop_run(const CoopRep& R, const CoopOps<T>& o, int x0, int y, int za, int n, T rr, int unit,
                                         double& qs) {
    constexpr int B = K * (int)sizeof(T);
    // rings of rows and of operands (the widest FP64 rows have registers for one operand plane only); FP64, bound by
    // its pipe, loses more to the instruction cache in a longer loop than it gains (128^3, N = 64: 4.46 ms
    // unrolled by 6, 4.18 by 2)
    constexpr int RU = sizeof(T) == 8 ? (B <= 16 ? 3 : 2) : B <= 8 ? 6 : B <= 12 ? 4 : B <= 16 || B > 24 ? 3 : 2, D = RU - 1;
    constexpr int EU = RU == 6 ? 3 : RU > 2 ? RU : B < 48 + 16 * (MODE == BLOCKED || MODE == BTILE) ? 2 : 1, DE = EU > 2 ? 2 : EU - 1;
    constexpr int UN = RU;
    constexpr bool SHIFT = UN % 3 != 0;   // the planes of the z pass move by copies
    const int lane = threadIdx.x & 31;
    const int nx = R.nx, ny = R.ny, nz = R.nz;
    const int plane = nx * ny;
    constexpr bool VEC = MODE == BLOCKED || MODE == BTILE || MODE == ROWS;
    // rows: this lane's row of the group (y), its place there; lanes past the group or past the last row idle
    const int lr = nx / K, grp = MODE == ROWS ? min(lane / lr, R.tile - 1) : 0, seg = grp * lr;
    const int yl = MODE == ROWS ? y * R.tile + grp : y;
    const bool on = MODE != ROWS || (yl < ny && lane < R.tile * lr);
    y = MODE == ROWS ? min(yl, ny - 1) : y;
    const int dm = (y == 0 ? ny - 1 : -1) * nx, dp = (y == ny - 1 ? 1 - ny : 1) * nx;   // to the y neighbours
    const int x1 = MODE == TILE || MODE == BTILE ? min(nx, x0 + R.tile) : nx;   // end of the outputs
    // lane's first column, its other columns, which of them exist
    const int LL = MODE == BLOCKED || MODE == ROWS ? lr - 1 : MODE == BTILE ? (x1 - x0) / K + 1 : 31;   // vectors: last lane
    const int li = min(lane - seg, LL);   // (only of VEC)
    int xl = VEC ? K * li : lane;
    if (MODE == BTILE) {
        xl += x0 - K;
        xl = xl < 0 ? xl + nx : (xl >= nx ? xl - nx : xl);
    }
    auto col = [&](int k) {   // relative to xl
        if (MODE != TILE) return 32 * k;
        int x = x0 - 1 + 32 * k + lane;
        return (x < 0 ? x + nx : (x >= nx ? x - nx : x)) - xl;
    };
    auto there = [&](int k) {   // loads: columns of the row (tile: up to the halo column of a ragged last tile)
        if (VEC) return true;
        if (MODE == STRIDED) return k < K - 1 || 32 * (K - 1) + lane < nx;
        return x0 - 1 + 32 * k + lane <= x1;
    };
    auto mine = [&](int k) {    // outputs
        if (MODE == BLOCKED) return lane <= LL;
        if (MODE == ROWS) return on;
        if (MODE == BTILE) return lane >= 1 && lane < LL;
        if (MODE == STRIDED) return k < K - 1 || 32 * (K - 1) + lane < nx;
        const int c = 32 * k + lane;
        return c >= 1 && x0 - 1 + c < x1;
    };
    auto get = [&](const T* p, T (&v)[K], bool outs) {
        if constexpr (VEC) {
            if (MODE != BTILE || !outs || mine(0)) ldk<T, K>(p, v);
        } else {
#pragma unroll
            for (int k = 0; k < K; ++k)
                if (outs ? mine(k) : there(k)) v[k] = p[col(k)];
        }
    };
    auto put = [&](T* p, const T (&v)[K]) {
        if constexpr (VEC) {
            if (mine(0)) stk<T, K>(p, v);
        } else {
#pragma unroll
            for (int k = 0; k < K; ++k)
                if (mine(k)) p[col(k)] = v[k];
        }
    };
    T raw[RU][3][K], e[EU][K], st[EU][K], q[EU][K], u[3][K];
#pragma unroll
    for (int k = 0; k < K; ++k) {   // (columns that do not exist stay 0)
#pragma unroll
        for (int d = 0; d < RU; ++d) raw[d][0][k] = raw[d][1][k] = raw[d][2][k] = T(0);
#pragma unroll
        for (int d = 0; d < EU; ++d) e[d][k] = st[d][k] = q[d][k] = T(0);
#pragma unroll
        for (int d = 0; d < 3; ++d) u[d][k] = T(0);
    }
    // sites (a field has fewer than 2^31) of the lane's first column: next plane to load, next output plane
    // to load operands of, output plane
    int zl = za == 0 ? nz - 1 : za - 1;
    int ol = zl * plane + y * nx + xl, oe = za * plane + y * nx + xl, ow = oe;
    auto load = [&](T (&v)[3][K]) {
        get(o.src + (ol + dm), v[0], false);
        get(o.src + ol, v[1], false);
        get(o.src + (ol + dp), v[2], false);
        ol += plane;
        if (++zl == nz) {
            zl = 0;
            ol -= nz * plane;
        }
    };
    auto loade = [&](int d) {
        get(o.E + oe, e[d], true);
        if constexpr (PAST) {
            get(o.st + oe, st[d], true);
            if (!o.first) get(o.q + oe, q[d], true);
        }
        oe += plane;
    };
    const int last = n + 2;
#pragma unroll
    for (int d = 0; d < D; ++d)
        if (d < last) load(raw[d]);
    const int lsrc = VEC ? seg + (li == 0 ? LL : li - 1) : ((lane + 31) & 31);
    const int rsrc = VEC ? seg + (li >= LL ? 0 : li + 1) : ((lane + 1) & 31);
    for (int i0 = 0; i0 < last; i0 += UN) {
#pragma unroll
        for (int d = 0; d < UN; ++d) {
            const int i = i0 + d;
            if (i >= last) break;
            if (i + D < last) load(raw[(d + D) % RU]);
            if ((d + DE >= 2 || i0 > 0) && i + DE < last) loade((d + DE) % EU);
            // y pass, then the x pass
            T t[K];
            T(&uc)[K] = u[SHIFT ? 2 : d % 3];
#pragma unroll
            for (int k = 0; k < K; ++k) t[k] = fma(rr, raw[d % RU][0][k] + raw[d % RU][2][k], raw[d % RU][1][k]);
            if constexpr (VEC) {   // (btile: wrong in the outer lanes, whose results are not used)
                const T lv = __shfl_sync(0xffffffffu, t[K - 1], lsrc), rv = __shfl_sync(0xffffffffu, t[0], rsrc);
#pragma unroll
                for (int k = 0; k < K; ++k)
                    uc[k] = fma(rr, (k ? t[k ? k - 1 : 0] : lv) + (k + 1 < K ? t[k + 1 < K ? k + 1 : k] : rv), t[k]);
            } else {
                T lf[K], rg[K];
#pragma unroll
                for (int k = 0; k < K; ++k) {
                    lf[k] = __shfl_sync(0xffffffffu, t[k], lsrc);
                    rg[k] = __shfl_sync(0xffffffffu, t[k], rsrc);
                }
                T lastv = lf[0], firstv = rg[0];
                const int ll = (nx - 1) & 31;              // lane of the row's last site (register K - 1)
                if constexpr (MODE == STRIDED) {
                    lastv = __shfl_sync(0xffffffffu, t[K - 1], ll);
                    firstv = __shfl_sync(0xffffffffu, t[0], 0);
                }
#pragma unroll
                for (int k = 0; k < K; ++k) {
                    const T l = lane > 0 ? lf[k] : (k > 0 ? lf[k > 0 ? k - 1 : 0] : lastv);
                    T r = lane < 31 ? rg[k] : rg[k < K - 1 ? k + 1 : k];
                    if (MODE == STRIDED && k == K - 1) r = lane == ll ? firstv : r;
                    uc[k] = fma(rr, l + r, t[k]);
                }
            }
            if (d >= 2 || i0 > 0) {
                constexpr int ring3 = 3;
                const int de = d % EU, um = SHIFT ? 0 : (d + 1) % ring3, u0 = SHIFT ? 1 : (d + 2) % ring3;
                T g[K], v[K];
#pragma unroll
                for (int k = 0; k < K; ++k) {
                    const T sg = fma(rr, u[um][k] + uc[k], u[u0][k]);
                    g[k] = e[de][k] * sg;
                    if constexpr (PAST) v[k] = fma(st[de][k], sg, q[de][k]);
                }
                if constexpr (PAST) put(o.q + ow, v);
                if (o.dst) put(o.dst + ow, g);
                ow += plane;
                if (PAST && o.lastQ) {
                    double qp = 0.0;
#pragma unroll
                    for (int k = 0; k < K; ++k)
                        if (mine(k)) qp += (double)g[k];
                    if (o.qrow) {
                        qp = warp_sum(qp);
                        if (lane == 0) o.qrow[unit + i - 2] = qp;
                    } else {
                        qs += qp;
                    }
                }
            }
            if constexpr (SHIFT) {
#pragma unroll
                for (int k = 0; k < K; ++k) {
                    u[0][k] = u[1][k];
                    u[1][k] = u[2][k];
                }
            }
        }
    }
}

// The first level of a chain, sigma[1] E (the passes' rounding included).
template <typename T, int K, int MODE>
__device__ __forceinline__ void coop_run_first(const CoopRep& R, const CoopOps<T>& o, int x0, int y, int za, int n, T rr) {
    const int lane = threadIdx.x & 31, nx = R.nx, plane = nx * R.ny;
    const T t = fma(rr, T(2), T(1)), u = fma(rr, t + t, t), sg = fma(rr, u + u, u);
    const int xe = MODE == TILE || MODE == BTILE ? min(nx, x0 + R.tile) : MODE == ROWS ? min(R.tile, R.ny - y * R.tile) * nx : nx;
    if (MODE == ROWS) y *= R.tile;   // (adjacent rows: one run of sites)
    for (int z = za; z < za + n; ++z)
        for (int x = x0 + lane; x < xe; x += 32) {
            const int i = z * plane + y * nx + x;
            o.dst[i] = o.E[i] * sg;
        }
}

// n planes from za of row y of x tile xt, at level j of chain C.
template <typename T, int K, int MODE, int C>
__device__ __forceinline__ void coop_rows(const CoopRep& R, const CoopOps<T>& o, int j, int xt, int y, int za, int n, double& qs) {
    const T rr = (T)R.rr;
    const int x0 = MODE == ROWS ? 0 : xt * R.tile;
    if (j == 0) coop_run_first<T, K, MODE>(R, o, x0, y, za, n, rr);
    else if (o.st) coop_run<T, K, MODE, true>(R, o, x0, y, za, n, rr, (xt * R.ny + y) * R.nz + za, qs);
    else coop_run<T, K, MODE, false>(R, o, x0, y, za, n, rr, 0, qs);
}

// Planes u0 .. u1 - 1 of the strips (strip-major) of a replica; of strips of 8 rows this warp's row.
template <typename T, int K, int MODE, int C>
__device__ __forceinline__ void coop_segment(const CoopRep& R, int j, int u0, int u1, int w, double& qs) {
    const CoopOps<T> o = coop_ops<T, C>(R, j);
    const int nz = R.nz;
    for (int u = u0; u < u1;) {
        const int g = u / nz, z = u - g * nz, n = min(nz - z, u1 - u);
        const int row = R.strip == 8 ? 8 * g + w : g;
        const int xt = MODE == TILE || MODE == BTILE ? row / R.ny : 0;
        coop_rows<T, K, MODE, C>(R, o, j, xt, row - xt * R.ny, z, n, qs);
        u += n;
    }
}

// The replicas' table in shared memory (the levels' acquire loads keep invalidating its cached copy): all of it,
// or, of more replicas than it holds, those from the first of the CTA's share on.
constexpr int kCoopShared = 128;
struct CoopTable {
    const CoopRep *loc, *all;   // shared, device
    int first;                  // the replica of loc[0]
    __device__ __forceinline__ const CoopRep& operator[](int i) const {
        return i - first < kCoopShared ? loc[i - first] : all[i];
    }
};

// This warp's share of a level.  KK: row layout of every replica of the launch, or 0: a switch per replica.
// cut: its run of the one replica (row; first plane, end), or the cost bounds of the warp and of its CTA.
struct CoopCut {
    int row, za, ze;
    int b0, b1, a0, a1;
    int r0;   // first replica of the CTA's share
};
template <typename T, int KK, int C>
__device__ __forceinline__ void coop_level(const CoopTable& tab, int nact, int runs, int j, int p, const CoopCut& cut) {
    if constexpr (KK > 0) {
        if (runs > 0) {
            const CoopRep& R = tab.loc[0];
            constexpr int MODE = (KK >> 4) - 1;
            double qs = 0.0;
            if (cut.za < cut.ze) {
                const int xt = MODE == TILE || MODE == BTILE ? cut.row / R.ny : 0;
                coop_rows<T, (KK & 15), MODE, C>(R, coop_ops<T, C>(R, j), j, xt, cut.row - xt * R.ny, cut.za, cut.ze - cut.za, qs);
            }
            if (C == 0 && j == R.N - 1 && !R.qrow) {   // s = N: this warp's share of Q
                const double t = warp_sum(qs);
                if ((threadIdx.x & 31) == 0) R.pq[p] = t;
            }
            return;
        }
    }
    const int w = threadIdx.x >> 5;
    for (int i = cut.r0; i < nact; ++i) {
        const CoopRep& R = tab[i];
        const int lay = KK > 0 ? KK : R.layout, wgt = R.wgt, planes = R.units / R.strip;
        const int b0 = R.strip == 8 ? cut.a0 : cut.b0, b1 = R.strip == 8 ? cut.a1 : cut.b1;
        const int c0 = R.cost0, c1 = c0 + planes * wgt;
        if (c1 <= cut.a0) continue;
        if (c0 >= cut.a1) break;
        // planes of the replica: cost bounds rounded up to whole planes
        const int u0 = b0 > c0 ? (b0 - c0 + wgt - 1) / wgt : 0;
        const int u1 = b1 < c1 ? (max(b1 - c0, 0) + wgt - 1) / wgt : planes;
        double qs = 0.0;
        if constexpr (KK > 0) {
            coop_segment<T, (KK & 15), (KK >> 4) - 1, C>(R, j, u0, u1, w, qs);
        } else {
#define DSCF_COOP_CASE(KV, MV) case KV + 16 * (MV + 1): coop_segment<T, KV, MV, C>(R, j, u0, u1, w, qs); break;
            switch (lay) {
                DSCF_COOP_LAYOUTS(DSCF_COOP_CASE)
                default: break;
            }
            if constexpr (sizeof(T) == 4) switch (lay) {
                DSCF_COOP_LAYOUTS32(DSCF_COOP_CASE)
                default: break;
            }
#undef DSCF_COOP_CASE
        }
        if (C == 0 && j == R.N - 1 && !R.qrow) {
            const double t = warp_sum(qs);
            if ((threadIdx.x & 31) == 0) R.pq[p] = t;
        }
    }
}

// Warps of a CTA, one CTA per SM: compute warps, and one warpgroup for the barriers, one warp per chain.
// Rows of at most 16 bytes a lane (FP32: 24) leave room for 12 compute warps of 160 registers a thread (the
// launch has 128: 12 x 160 + 4 x 24 <= 16 x 128), longer ones for 8 of 232 (168: 8 x 232 + 4 x 24 <= 12 x
// 168).  N = 32, FP32, 8 and 12 warps: 140 x 80 x 80 274 and 265 us, 163 x 80 x 80 303 and 291, but 200 x
// 100 x 64 323 and 371, 256^3 3.92 and 4.08 ms.
constexpr int kCoopSync = 4, kCoopSyncRegs = 24;
template <int NW>
constexpr int kCoopRegs = NW == 12 ? 160 : 232;
template <typename T>
__host__ __device__ constexpr int coop_nw(int kk) { return coop_warps(kk, sizeof(T) == 8); }

__device__ __forceinline__ void bar_wait(unsigned long long* bar, unsigned parity, const CoopCtl& ctl, bool& dead) {
    if (dead) return;
    for (long long spins = 0; !bar_test(bar, parity); ++spins)
        if (spins > kBarSpinLimit) {
            atomicOr(ctl.status, (int)ST_TIMEOUT);
            atomicExch(ctl.abort, 1);
            dead = true;
            return;
        }
}

template <typename T, int KK>
__global__ void __launch_bounds__(32 * (coop_nw<T>(KK) + kCoopSync), 1) k_prop_coop(const CoopCtl ctl) {
    constexpr int NW = coop_nw<T>(KK);
    __shared__ CoopRep tab[kCoopShared];
    __shared__ __align__(8) unsigned long long done[2], go[2];   // per chain: level computed here; computed everywhere
    __shared__ bool fin;
    const int ncta = (int)gridDim.x, w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const bool sync = ctl.j1 - ctl.j0 > 1;   // one level per launch: the launches are the barriers
    const CoopRep* reps = ctl.nrep <= kCoopShared ? tab : ctl.reps;
    constexpr int WORDS = sizeof(CoopRep) / sizeof(int);
    if (ctl.nrep <= kCoopShared) {
        for (int i = threadIdx.x; i < ctl.nrep * WORDS; i += blockDim.x) ((int*)tab)[i] = ((const int*)ctl.reps)[i];
    }
    if (threadIdx.x == 0) {
        for (int c = 0; c < 2; ++c) {
            bar_init(&done[c], NW);
            bar_init(&go[c], 1);
        }
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    __syncthreads();
    bool dead = false;
    if (w >= NW) {
        // ---- barrier warps, one per chain: the compute warps go on with the other chain meanwhile ----
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;\n" ::"n"(kCoopSyncRegs));
        const int c = w - NW;
        if (!sync || c >= 2 || lane != 0) return;
        bool aborted = ld_acquire(ctl.abort) != 0;
        int* f = ctl.cnt + c * kFlagStride;
        for (int d = 0; d < ctl.j1 - ctl.j0; ++d) {
            bar_wait(&done[c], (unsigned)(d & 1), ctl, dead);
            // `done` orders the compute warps' stores before this release; release is cumulative
            red_release(f);
            const int target = (d + 1) * ncta;
            int spins = 0;
            while (!aborted && ld_acquire(f) < target) {
                if ((++spins & 31) == 0) {
                    if (ld_acquire(ctl.abort) != 0) {
                        aborted = true;
                    } else if (spins > ctl.limit) {
                        atomicOr(ctl.status, (int)ST_TIMEOUT);
                        atomicExch(ctl.abort, 1);
                        aborted = true;
                    }
                }
                __nanosleep(20);
            }
            bar_arrive(&go[c]);
        }
        // the last of all barrier warps leaves the counters at zero
        __threadfence();
        if (atomicInc((unsigned*)ctl.cnt + 2 * kFlagStride, 2u * (unsigned)ncta - 1u) == 2u * (unsigned)ncta - 1u) {
            ctl.cnt[0] = 0;
            ctl.cnt[kFlagStride] = 0;
        }
        return;
    }
    // ---- compute warps ----
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;\n" ::"n"(kCoopRegs<NW>));
    const int p = blockIdx.x * NW + w;
    int nact = ctl.nrep + 1;        // active replicas
    int ends = 0;                   // the level after the shortest active chain's last
    CoopTable table = {tab, ctl.reps, 0};
    CoopCut cut = {};
    if (ctl.runs > 0) {
        const CoopRep& R = reps[0];
        const int i = blockIdx.x * ctl.per + w, k = i % ctl.runs;
        cut.row = i / ctl.runs;
        if (w < ctl.per && cut.row * R.nz < R.units) {
            cut.za = (int)((long long)R.nz * k / ctl.runs);
            cut.ze = (int)((long long)R.nz * (k + 1) / ctl.runs);
        }
    }
    if (ctl.j0 == 0) {   // shares of Q of replicas this warp has none of
        for (int r = lane; r < ctl.nrep; r += 32)
            if (!reps[r].qrow) reps[r].pq[p] = 0.0;
        __syncwarp();
    }
    for (int j = ctl.j0; j < ctl.j1; ++j) {
        const int before = nact;
        if (j >= ends) {
            nact = min(nact, ctl.nrep);
            while (reps[nact - 1].N <= j) --nact;   // (the longest chain has more levels)
            ends = reps[nact - 1].N;
        }
        if (nact != before) {
            const CoopRep& last = reps[nact - 1];
            const long long total = last.cost0 + last.units / last.strip * last.wgt;
            const long long P = ncta * NW, pa = blockIdx.x * NW;
            cut.b0 = (int)(total * p / P);
            cut.b1 = (int)(total * (p + 1) / P);
            cut.a0 = (int)(total * pa / P);
            cut.a1 = (int)(total * (pa + NW) / P);
            // the last replica that begins at a0 or before (all of them at every level, and their sums of Q all
            // in the first CTAs below: a step of five evaluations of 200 replicas of 8^3 sites, N = 8, FP32 4241
            // us, 557 so, 602 with a launch per level; 40 of 20^3, N = 16, 1438, 804, 1106)
            int lo = 0, hi = nact - 1;
            while (lo < hi) {
                const int m = (lo + hi + 1) >> 1;
                if (reps[m].cost0 <= cut.a0) lo = m;
                else hi = m - 1;
            }
            cut.r0 = lo;
            if (ctl.nrep > kCoopShared) {
                asm volatile("bar.sync 1, %0;\n" ::"r"(32 * NW) : "memory");   // every warp is done with the table's last part
                const int n = min(kCoopShared, nact - lo) * WORDS;
                for (int i = threadIdx.x; i < n; i += 32 * NW) ((int*)tab)[i] = ((const int*)(ctl.reps + lo))[i];
                asm volatile("bar.sync 1, %0;\n" ::"r"(32 * NW) : "memory");
                table.first = lo;
            }
        }
        const int d = j - ctl.j0;            // levels of this launch before this one
        const unsigned par = (unsigned)((d - 1) & 1);
        if (sync && d > 0) {
            bar_wait(&go[0], par, ctl, dead);
            // another cut of the work when chains end: what a warp has written itself so far may now
            // be another warp's, so both chains' levels must be complete
            if (nact != before) bar_wait(&go[1], par, ctl, dead);
            __syncwarp();
        }
        coop_level<T, KK, 0>(table, nact, ctl.runs, j, p, cut);
        if (sync) {
            __syncwarp();
            if (lane == 0) bar_arrive(&done[0]);
            if (d > 0) bar_wait(&go[1], par, ctl, dead);
            __syncwarp();
        }
        coop_level<T, KK, 1>(table, nact, ctl.runs, j, p, cut);
        if (sync) {
            __syncwarp();
            if (lane == 0) bar_arrive(&done[1]);
        }
    }
    if (sync) {
        // Q: every 32 row planes of a replica make one partial sum, whatever the cut of the work, so a
        // replica's Q is the same alone and in any batch
        bar_wait(&go[0], (unsigned)((ctl.j1 - ctl.j0 - 1) & 1), ctl, dead);
        __syncwarp();
        // (replica r's from the r-th CTA on, so that many small replicas do not all meet in the first)
        const int P = ncta * NW;
        for (int rb = 0; rb < ctl.nrep; rb += 32) {
            const int r = rb + lane;
            int g0 = 0;
            bool some = false;
            if (r < ctl.nrep) {
                g0 = p - r % ncta * NW;
                g0 += g0 < 0 ? P : 0;
                some = 32LL * g0 < reps[r].units;
            }
            for (unsigned m = __ballot_sync(0xffffffffu, some); m; m &= m - 1) {
                const int k = __ffs(m) - 1;
                const CoopRep& R = reps[rb + k];
                const int units = R.units;
                for (int g = __shfl_sync(0xffffffffu, g0, k); 32LL * g < units; g += P) {
                    const int u = 32 * g + lane;
                    const double t = warp_sum(u < units ? R.qrow[u] : 0.0);
                    if (lane == 0) R.pq[g] = t;
                }
            }
        }
        // the last CTA adds up the partial sums, in order
        asm volatile("bar.sync 1, %0;\n" ::"r"(32 * NW) : "memory");
        if (threadIdx.x == 0) {
            __threadfence();
            fin = atomicInc((unsigned*)ctl.cnt + 2 * kFlagStride + 16, (unsigned)ncta - 1u) == (unsigned)ncta - 1u;
        }
        asm volatile("bar.sync 1, %0;\n" ::"r"(32 * NW) : "memory");
        if (fin) {
            __threadfence();
            constexpr int U = 4;   // replicas of a warp side by side: their loads' latencies overlap
            for (int r = w; r < ctl.nrep; r += U * NW) {
                double s[U];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    s[u] = 0.0;
                    if (r + u * NW >= ctl.nrep) continue;
                    const CoopRep& R = reps[r + u * NW];
                    for (int g = lane; 32LL * g < R.units; g += 32) s[u] += __ldcg(R.pq + g);
                }
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    if (r + u * NW >= ctl.nrep) break;
                    double* q = reps[r + u * NW].qsum;
                    if constexpr (sizeof(T) == 8) {
                        const Two t = warp_sum(Two{s[u], 0.0});
                        if (lane == 0) {
                            q[0] = t.hi;
                            q[S_QLO - S_QSUM] = t.lo;
                        }
                    } else {
                        const double t = warp_sum(s[u]);
                        if (lane == 0) *q = t;
                    }
                }
            }
        }
    }
}

template <typename T>
const void* coop_kernel(int kk) {
#define DSCF_COOP_KERNEL(KV, MV) case KV + 16 * (MV + 1): return (const void*)k_prop_coop<T, KV + 16 * (MV + 1)>;
    if constexpr (sizeof(T) == 4) switch (kk) {
        DSCF_COOP_LAYOUTS32(DSCF_COOP_KERNEL)
        default: break;
    }
    switch (kk) {
        DSCF_COOP_LAYOUTS(DSCF_COOP_KERNEL)
        default: return coop_mixed<T>();
    }
#undef DSCF_COOP_KERNEL
}

}  // namespace

// Checks that the kernels launch with the registers their warps share out (setmaxnreg would wait for
// ever if they did not).
template <typename T>
int coop_prepare(int kk) {
    const int nw = coop_nw<T>(kk);
    cudaFuncAttributes fa;
    cudaError_t e = cudaFuncGetAttributes(&fa, coop_kernel<T>(kk));
    if (e == cudaSuccess && fa.numRegs * (nw + kCoopSync) < (nw == 12 ? kCoopRegs<12> : kCoopRegs<8>) * nw + kCoopSyncRegs * kCoopSync)
        e = cudaErrorInvalidConfiguration;
    return (int)e;
}

template <typename T>
int launch_prop_coop(const Launch& L, const CoopPlan& c, int j0, int j1, int limit) {
    CoopCtl ctl;
    ctl.reps = c.reps;
    ctl.nrep = c.nrep;
    ctl.j0 = j0;
    ctl.j1 = j1;
    ctl.cnt = c.cnt;
    ctl.abort = c.abort;
    ctl.status = L.status;
    ctl.limit = limit;
    ctl.runs = c.runs;
    ctl.per = c.per;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(c.ncta);
    cfg.blockDim = dim3(32 * (coop_nw<T>(c.kk) + kCoopSync));
    cfg.stream = L.stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = j1 - j0 > 1 ? 1 : 0;
    void* args[] = {(void*)&ctl};
    return (int)cudaLaunchKernelExC(&cfg, coop_kernel<T>(c.kk), args);
}

}  // namespace dscf
