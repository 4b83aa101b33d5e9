// Learned predictor of the density map: a translation-invariant 3-D convolution network
// phi_hat_I = phibar_I + y_I - <y_I>,  y = conv3(tanh(conv2(tanh(conv1(U - <U>))))),
// circular 5^3 kernels, 2 -> 32 -> 32 -> 2 channels (the paper has no such component; it stands
// in for the propagator solve inside the self-consistent inversion).
//
// Tensor cores: every convolution (forward, and backward with respect to the input) is one
// implicit GEMM over (offset, input channel) in BF16 with FP32 accumulation; weight gradients are
// per-offset GEMMs over sites.  The forward convolutions run on tcgen05 (operands in shared
// memory, accumulators in tensor memory; dscf_tc.cu) when nx is a multiple of 128 and ny of 8,
// and with warp-level mma.sync m16n8k16 on input blocks staged in shared memory otherwise (and for
// the backward pass).  Activations are stored
// channel-last in BF16 with channel counts padded to multiples of 16 (zero weights in the pad);
// the tcgen05 forward keeps its own copies in a padded channel-group layout (x16f, h1p, h2p) from
// which it stages rows by bulk copies, and the backward pass reads channel-last copies of them.
// Training keeps FP32 master weights and Adam moments.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cmath>
#include <cstring>
#include <new>
#include <string>
#include <type_traits>
#include <vector>

#include "../../include/dscf.h"
#include "dscf_internal.cuh"

using namespace dscf;

namespace {

typedef __nv_bfloat16 bf16;

constexpr int NL = 3;
constexpr int KVOL = 125;
constexpr int CIN[NL] = {2, 32, 32}, COUT[NL] = {32, 32, 2};
constexpr int CINP[NL] = {16, 32, 32}, COUTP[NL] = {32, 32, 16};
constexpr int NTF[NL] = {4, 4, 1};   // n-tiles of 8 output channels of the mma.sync forward
constexpr size_t wcount(int l) { return (size_t)COUT[l] * CIN[l] * KVOL; }
constexpr size_t NPARAM = wcount(0) + 32 + wcount(1) + 32 + wcount(2) + 2;

enum { EPI_TANH = 0, EPI_LIN_F32 = 1, EPI_DTANH = 2 };

__device__ __forceinline__ unsigned pack2(bf16 lo, bf16 hi) {
    return (unsigned)__bfloat16_as_ushort(lo) | ((unsigned)__bfloat16_as_ushort(hi) << 16);
}
__device__ __forceinline__ void mma16816(float* c, const unsigned* a, const unsigned* b) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};\n"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}
__device__ __forceinline__ unsigned sm_addr(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void ldsm4(unsigned addr, unsigned (&r)[4]) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
__device__ __forceinline__ void ldsm4t(unsigned addr, unsigned (&r)[4]) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
__device__ __forceinline__ void cp_async16(unsigned dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(dst), "l"(src));
}
// the same, zeros instead of the source where !ok
__device__ __forceinline__ void cp_async16z(unsigned dst, const void* src, bool ok) {
    const int n = ok ? 16 : 0;
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(dst), "l"(src), "r"(n));
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory"); }

// Byte offset of 16-byte chunk c (8 channels) of staged site i, C channels per site: chunks are
// permuted within 128-byte lines so that the 8 consecutive sites of an ldmatrix row group fall
// into different banks.
template <int C>
__device__ __forceinline__ unsigned swz(int i, int c) {
    if constexpr (C == 32) return (unsigned)(i * 64 + ((c ^ ((i >> 1) & 3)) << 4));
    else return (unsigned)(i * 32 + ((c ^ ((i >> 2) & 1)) << 4));
}

// Implicit-GEMM circular 5^3 convolution on mma.sync:
//   out[r][co] = sum_o sum_ci in[r + o][ci] W[o][co][ci]  (+ epilogue)
// in: [B][V][CI] bf16; W: fragments (k_prep_w).  A CTA of four warps computes a block of 16 MX x 4 x
// (4 / MX) sites whose input, two sites larger on every side, it stages once in shared memory; a
// warp holds four m-tiles of 16 sites, so an offset's weight fragments (16-byte loads in fragment
// order, fetched an offset ahead) serve four tiles and an input fragment is one ldmatrix.  Blocks of
// two tiles in x for rows of a multiple of 32 sites (fewest halo sites), of one otherwise; two CTAs
// per SM (32 input channels: 110 KB each), so one stages while the other computes.
// Tensor-pipe bound: per offset a warp issues 4 x 2 x 4 MMAs against 8 ldmatrix (32 -> 32 channels:
// 8 x 32^3 sites in 240 us = 280 TFLOP/s; 32 -> 8: 167 us, ldmatrix bound; before, with 4-byte
// gathers from global memory and no reuse of weights, a gradient's five convolutions took 2.4 ms).
// Each accumulator takes its products in the order (offset, channel group).
// Epilogues: tanh(acc + bias) -> bf16; acc + bias -> f32 (channels 0 and 1 of 16 stored per site);
// acc * (1 - h^2) with h the forward activation -> bf16, with bgrad != NULL also summed per channel
// into bgrad in FP32: the bias gradient of the layer whose activation is hact.
constexpr int CV_TY = 4;
template <int MX>
struct ConvTile {
    static constexpr int TZ = 4 / MX, HX = 16 * MX + 4, HY = CV_TY + 4, HZ = TZ + 4, SITES = HX * HY * HZ;
};
template <int CI, int NT, int EPI, int MX>
__global__ void __launch_bounds__(128, CI == 32 ? 2 : 3) k_conv(const bf16* __restrict__ in, const uint4* __restrict__ W,
                                                                const float* __restrict__ bias, int cout,
                                                                const bf16* __restrict__ hact, void* __restrict__ out,
                                                                int nx, int ny, int nz, float* __restrict__ bgrad) {
    using CT = ConvTile<MX>;
    constexpr int HX = CT::HX, HY = CT::HY, KC = CI / 16, CO = NT == 1 ? 16 : NT * 8;
    constexpr int WV = KC * NT / 2;            // 16-byte weight vectors per lane and offset
    extern __shared__ __align__(128) unsigned char smem[];
    const unsigned sm0 = sm_addr(smem);
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int V = nx * ny * nz;
    // block -> sample, origin
    int t = blockIdx.x;
    const int nbx = nx / (16 * MX), nby = (ny + CV_TY - 1) / CV_TY, nbz = (nz + CT::TZ - 1) / CT::TZ;
    const int x0 = (t % nbx) * 16 * MX;
    t /= nbx;
    const int y0 = (t % nby) * CV_TY;
    t /= nby;
    const int z0 = (t % nbz) * CT::TZ, b = t / nbz;
    const bf16* inb = in + (size_t)b * V * CI;
    constexpr int CPS = CI / 8;                // 16-byte chunks per site
    for (int i = tid; i < CT::SITES * CPS; i += 128) {
        const int site = i / CPS, c = i - site * CPS;
        const int hx = site % HX, hyz = site / HX, hy = hyz % HY, hz = hyz / HY;
        int x = x0 + hx - 2, y = y0 + hy - 2, z = z0 + hz - 2;
        x = x < 0 ? x + nx : (x >= nx ? x - nx : x);
        y = (y % ny + ny) % ny;                // ragged blocks reach further than one wrap
        z = (z % nz + nz) % nz;
        cp_async16(sm0 + swz<CI>(site, c), inb + (size_t)((z * ny + y) * nx + x) * CI + c * 8);
    }
    cp_async_commit();
    const uint4* wl = W + lane * WV;
    uint4 wn[WV];
#pragma unroll
    for (int v = 0; v < WV; ++v) wn[v] = __ldg(wl + v);
    float acc[4][NT][4];
#pragma unroll
    for (int m = 0; m < 4; ++m)
#pragma unroll
        for (int j = 0; j < NT; ++j) acc[m][j][0] = acc[m][j][1] = acc[m][j][2] = acc[m][j][3] = 0.f;
    cp_async_wait<0>();
    __syncthreads();
    // this warp's tiles: MX = 2: plane w / 2, rows 2 (w % 2) + m / 2, x half m % 2; MX = 1: plane w, row m
    const int wz = MX == 2 ? w >> 1 : w, wy = MX == 2 ? 2 * (w & 1) : 0;
    const int row = (lane & 7) + ((lane >> 3) & 1) * 8, ch = lane >> 4;
    int o = 0;
#pragma unroll 1
    for (int ozy = 0; ozy < 25; ++ozy) {
        const int i0 = ((wz + ozy / 5) * HY + wy + ozy % 5) * HX + row;
#pragma unroll
        for (int ox = 0; ox < 5; ++ox, ++o) {
            unsigned wf[WV * 4];
#pragma unroll
            for (int v = 0; v < WV; ++v) {
                wf[4 * v] = wn[v].x; wf[4 * v + 1] = wn[v].y; wf[4 * v + 2] = wn[v].z; wf[4 * v + 3] = wn[v].w;
            }
            if (o + 1 < KVOL) {
#pragma unroll
                for (int v = 0; v < WV; ++v) wn[v] = __ldg(wl + (size_t)(o + 1) * 32 * WV + v);
            }
            const unsigned base = swz<CI>(i0 + ox, ch);   // tile 0
#pragma unroll
            for (int kc = 0; kc < KC; ++kc) {
                // the other tiles lie a constant number of sites on; a row (HX sites) later the chunk
                // permutation differs by one fixed bit (HX = 36 or 20), 16 sites later it is the same
                unsigned a[4][4];
#pragma unroll
                for (int m = 0; m < 4; ++m) {
                    const int dr = MX == 2 ? m >> 1 : m, di = dr * HX + (MX == 2 ? 16 * (m & 1) : 0);
                    const unsigned flip = (dr & 1) ? (CI == 32 ? 32u : 16u) : 0u;
                    ldsm4(sm0 + ((base + di * CI * 2) ^ flip ^ (kc ? 32u : 0u)), a[m]);
                }
#pragma unroll
                for (int j = 0; j < NT; ++j)
#pragma unroll
                    for (int m = 0; m < 4; ++m) mma16816(acc[m][j], a[m], wf + (kc * NT + j) * 2);
            }
        }
    }
    // epilogue: rows g, g + 8 of each tile, columns co = 8 j + 2 t, + 1
    const int g = lane >> 2, tq = lane & 3;
#pragma unroll
    for (int j = 0; j < NT; ++j) {
        const int co = j * 8 + 2 * tq;
        const float b0 = (EPI != EPI_DTANH && co < cout) ? bias[co] : 0.f;
        const float b1 = (EPI != EPI_DTANH && co + 1 < cout) ? bias[co + 1] : 0.f;
        float bs0 = 0.f, bs1 = 0.f;
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            const int y = y0 + wy + (MX == 2 ? m >> 1 : m), z = z0 + wz;
            if (y >= ny || z >= nz) continue;
            const size_t s0 = (size_t)b * V + (size_t)(z * ny + y) * nx + x0 + (MX == 2 ? 16 * (m & 1) : 0) + g;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const size_t site = s0 + 8 * h;
                float v0 = acc[m][j][2 * h] + b0, v1 = acc[m][j][2 * h + 1] + b1;
                if (EPI == EPI_TANH) {
                    v0 = tanhf(v0);
                    v1 = tanhf(v1);
                    *(unsigned*)((bf16*)out + site * CO + co) = pack2(__float2bfloat16(v0), __float2bfloat16(v1));
                } else if (EPI == EPI_LIN_F32) {
                    if (tq == 0) *(float2*)((float*)out + site * CO) = make_float2(v0, v1);
                } else {
                    v0 = acc[m][j][2 * h];
                    v1 = acc[m][j][2 * h + 1];
                    const __nv_bfloat162 hh = *(const __nv_bfloat162*)(hact + site * CO + co);
                    const float h0 = __low2float(hh), h1 = __high2float(hh);
                    v0 *= 1.f - h0 * h0;
                    v1 *= 1.f - h1 * h1;
                    bs0 += v0;
                    bs1 += v1;
                    *(unsigned*)((bf16*)out + site * CO + co) = pack2(__float2bfloat16(v0), __float2bfloat16(v1));
                }
            }
        }
        if (EPI == EPI_DTANH && bgrad) {   // sum over the 8 row groups (lane bits 2..4)
#pragma unroll
            for (int s = 4; s < 32; s <<= 1) {
                bs0 += __shfl_xor_sync(0xffffffffu, bs0, s);
                bs1 += __shfl_xor_sync(0xffffffffu, bs1, s);
            }
            if (g == 0) {
                if (co < cout) atomicAdd(&bgrad[co], bs0);
                if (co + 1 < cout) atomicAdd(&bgrad[co + 1], bs1);
            }
        }
    }
}

// Weight gradient of one layer: dW[co][ci][o] = sum_r in[r + o][ci] dout[r][co], a GEMM per offset
// (M = input channels, N = output channels, K = sites) on mma.sync.  A CTA keeps the 25 offsets of one
// dz in registers, spread over 12 warps (three per tensor core: 2 offsets each, the last warp 3; CI x
// 8 NT accumulators per offset over the lanes), and goes over every nsplit-th tile of 8 rows x 16 MX
// sites: per tile it stages the rows of dout and the rows of in at plane z + dz, two larger in y
// and x, in one of two shared-memory buffers while it computes from the other, so a staged site is
// used by 25 offsets and a dout fragment by a warp's two.  Per 16 sites a warp issues 2 x 2 x 4 MMAs
// against 6 ldmatrix (32 x 32 channels): tensor-pipe bound.  The tensor core truncates its sums, so
// a long chain of MMAs drifts (560 of them: 2e-5 of the gradient); every second tile the accumulators
// are added, rounded, to the CTA's totals in shared memory and start again (32 MMAs: 1e-6).  The
// totals of a CTA go to part[split][o][CI][8 NT]; k_wgrad_sum adds the splits in order.  8 x 32^3
// sites: 230 us (32 x 32), 147 and 142 us (32 x 2, 2 x 32); 3.9 ms together with 2-byte gathers and
// atomics per 128 sites.
constexpr int WG_TY = 8, WG_WARPS = 12, WG_OFF = 3;   // rows per tile; warps; most offsets per warp
constexpr int WG_FLUSH = 2;                             // tiles between additions to the totals
template <int CI, int NT, int CD, int MX>
struct WgTile {
    static constexpr int HX = 16 * MX + 4, HY = WG_TY + 4;
    static constexpr int INB = HX * HY * CI * 2, DB = 16 * MX * WG_TY * CD * 2;   // bytes staged of in and dout
    static constexpr int SMEM = 2 * (INB + DB) + 25 * CI * 8 * NT * 4;
};
template <int CI, int NT, int CD, int MX>   // CD: channels per site of dout
__global__ void __launch_bounds__(32 * WG_WARPS, 1) k_wgrad(const bf16* __restrict__ in, const bf16* __restrict__ dout,
                                                            float* __restrict__ part, int nx, int ny, int nz, int B) {
    using WT = WgTile<CI, NT, CD, MX>;
    constexpr int HX = WT::HX, HY = WT::HY, TX = 16 * MX, MI = CI / 16, T = 32 * WG_WARPS;
    extern __shared__ __align__(128) unsigned char smem[];
    const unsigned sm0 = sm_addr(smem);
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int split = blockIdx.x, nsplit = gridDim.x, dz = blockIdx.y;
    const int nbx = nx / TX, nby = (ny + WG_TY - 1) / WG_TY;
    const int ntile = B * nz * nby * nbx;
    const size_t V = (size_t)nx * ny * nz;
    auto stage = [&](int tile, int buf) {
        int t = tile;
        const int x0 = (t % nbx) * TX;
        t /= nbx;
        const int y0 = (t % nby) * WG_TY;
        t /= nby;
        const int z = t % nz, b = t / nz;
        const int zi = ((z + dz - 2) % nz + nz) % nz;
        const unsigned si = sm0 + buf * (WT::INB + WT::DB), sd = si + WT::INB;
        const bf16* inb = in + ((size_t)b * V + (size_t)zi * ny * nx) * CI;
        for (int i = tid; i < HX * HY * (CI / 8); i += T) {
            const int site = i / (CI / 8), c = i - site * (CI / 8);
            const int hx = site % HX, hy = site / HX;
            int x = x0 + hx - 2;
            x = x < 0 ? x + nx : (x >= nx ? x - nx : x);
            const int y = ((y0 + hy - 2) % ny + ny) % ny;
            cp_async16(si + swz<CI>(site, c), inb + (size_t)(y * nx + x) * CI + c * 8);
        }
        const bf16* db = dout + ((size_t)b * V + (size_t)z * ny * nx) * CD;
        for (int i = tid; i < TX * WG_TY * (CD / 8); i += T) {
            const int site = i / (CD / 8), c = i - site * (CD / 8);
            const int x = x0 + site % TX, y = y0 + site / TX;
            cp_async16z(sd + swz<CD>(site, c), db + (size_t)((y < ny ? y : 0) * nx + x) * CD + c * 8, y < ny);   // rows past ny add nothing
        }
        cp_async_commit();
    };
    float acc[WG_OFF][MI][NT][4];
#pragma unroll
    for (int o = 0; o < WG_OFF; ++o)
#pragma unroll
        for (int i = 0; i < MI; ++i)
#pragma unroll
            for (int j = 0; j < NT; ++j) acc[o][i][j][0] = acc[o][i][j][1] = acc[o][i][j][2] = acc[o][i][j][3] = 0.f;
    const int o0 = 2 * w, no = w == WG_WARPS - 1 ? 3 : 2;   // offsets o0 .. o0 + no - 1 of the plane's 25
    // ldmatrix rows: in: sites k (lane & 7, + 8 for the upper lane half), channel chunk by lane bit 3;
    // dout: sites k by lane bits 0-3, chunk by lane bit 4
    const int ka = (lane & 7) + ((lane >> 4) << 3), ca = (lane >> 3) & 1;
    const int kb = lane & 15, cb = lane >> 4;
    int doff[WG_OFF];   // site shift of each offset
#pragma unroll
    for (int o = 0; o < WG_OFF; ++o) doff[o] = (o0 + o) / 5 * HX + (o0 + o) % 5 + ka;
    // the thread's totals: value pairs (offset, m-tile, n-tile, row half), 32 lanes side by side
    float2* tot = (float2*)(smem + 2 * (WT::INB + WT::DB)) + o0 * (CI * 4 * NT) + lane;
    int left = WG_FLUSH;
    bool first = true;
    auto flush = [&]() {
#pragma unroll
        for (int o = 0; o < WG_OFF; ++o) {
            if (o >= no) break;
#pragma unroll
            for (int i = 0; i < MI; ++i)
#pragma unroll
                for (int j = 0; j < NT; ++j)
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        float2* q = tot + (((o * MI + i) * NT + j) * 2 + h) * 32;
                        float2 v = make_float2(acc[o][i][j][2 * h], acc[o][i][j][2 * h + 1]);
                        if (!first) {
                            const float2 u = *q;
                            v.x += u.x;
                            v.y += u.y;
                        }
                        *q = v;
                        acc[o][i][j][2 * h] = acc[o][i][j][2 * h + 1] = 0.f;
                    }
        }
        first = false;
        left = WG_FLUSH;
    };
    int buf = 0;
    if (split < ntile) stage(split, 0);
    for (int tile = split; tile < ntile; tile += nsplit, buf ^= 1) {
        if (tile + nsplit < ntile) {
            stage(tile + nsplit, buf ^ 1);
            cp_async_wait<1>();
        } else {
            cp_async_wait<0>();
        }
        __syncthreads();
        const unsigned si = sm0 + buf * (WT::INB + WT::DB), sd = si + WT::INB;
#pragma unroll 2
        for (int ks = 0; ks < WG_TY * MX; ++ks) {
            const int r = ks / MX, xs = (ks % MX) * 16;
            unsigned bf[(NT + 1) / 2][4];
#pragma unroll
            for (int jp = 0; jp < (NT + 1) / 2; ++jp) ldsm4t(sd + swz<CD>(r * TX + xs + kb, jp * 2 + cb), bf[jp]);
#pragma unroll
            for (int o = 0; o < WG_OFF; ++o) {
                if (o == 2 && no < 3) break;   // uniform in the warp
                const int site = r * HX + xs + doff[o];
#pragma unroll
                for (int i = 0; i < MI; ++i) {
                    unsigned a[4];
                    ldsm4t(si + swz<CI>(site, 2 * i + ca), a);
#pragma unroll
                    for (int j = 0; j < NT; ++j) mma16816(acc[o][i][j], a, &bf[j >> 1][(j & 1) * 2]);
                }
            }
        }
        if (--left == 0) flush();
        __syncthreads();   // the buffer is staged over after the next tile
    }
    flush();
    // rows = input channel (g, g + 8 within the m-tile), columns = output channel (2 t, 2 t + 1)
    const int g = lane >> 2, tq = lane & 3;
    float* p = part + ((size_t)split * KVOL + dz * 25 + o0) * (CI * 8 * NT);
    for (int o = 0; o < no; ++o)
#pragma unroll
        for (int i = 0; i < MI; ++i)
#pragma unroll
            for (int j = 0; j < NT; ++j)
#pragma unroll
                for (int h = 0; h < 2; ++h)
                    *(float2*)(p + (size_t)o * (CI * 8 * NT) + (i * 16 + g + 8 * h) * (8 * NT) + j * 8 + 2 * tq) =
                        tot[(((o * MI + i) * NT + j) * 2 + h) * 32];
}
// dW[co][ci][o] = sum over the splits of part[split][o][CI][CO8], in order; one thread per (o, ci, co).
__global__ void __launch_bounds__(256) k_wgrad_sum(const float* __restrict__ part, int nsplit, int CI, int CO8, int cin,
                                                   int cout, float* __restrict__ dW) {
    const int n = KVOL * CI * CO8;
    const int i = blockIdx.x * 256 + threadIdx.x;
    if (i >= n) return;
    const int co = i % CO8, ci = i / CO8 % CI, o = i / (CO8 * CI);
    if (co >= cout || ci >= cin) return;
    float s = 0.f;
#pragma unroll 8
    for (int k = 0; k < nsplit; ++k) s += part[(size_t)k * n + i];
    dW[((size_t)co * cin + ci) * KVOL + o] = s;
}

// Per-sample, per-channel FP64 partial sums of a [B][C][V] float field (grid: blocks x C x B).  WIDE: a
// thread takes several sites and sums them in FP64 (grids of few sites, where a block per 256 sites
// would be mostly launch cost: 27 us for 8 x 32^3, 4 us with 4096 sites per block).
template <bool WIDE>
__global__ void k_chan_parts(const float* __restrict__ f, int C, int V, double* __restrict__ part) {
    __shared__ double sh[33];
    const int c = blockIdx.y, b = blockIdx.z;
    const float* p = f + ((size_t)b * C + c) * V;
    std::conditional_t<WIDE, double, float> acc = 0;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < V; i += gridDim.x * blockDim.x) acc += p[i];
    const double t = block_sum((double)acc, sh);
    if (threadIdx.x == 0) part[((size_t)b * C + c) * gridDim.x + blockIdx.x] = t;
}
// Same for a channel-last [B][V][CS] float field (channels 0..C-1).
template <bool WIDE>
__global__ void k_chan_parts_cl(const float* __restrict__ f, int C, int CS, int V, double* __restrict__ part) {
    __shared__ double sh[33];
    const int c = blockIdx.y, b = blockIdx.z;
    const float* p = f + (size_t)b * V * CS + c;
    std::conditional_t<WIDE, double, float> acc = 0;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < V; i += gridDim.x * blockDim.x) acc += p[(size_t)i * CS];
    const double t = block_sum((double)acc, sh);
    if (threadIdx.x == 0) part[((size_t)b * C + c) * gridDim.x + blockIdx.x] = t;
}
// means[p] = (sum of the nb partials of pair p, fixed order) / V, one block per pair.
__global__ void k_chan_final(const double* __restrict__ part, int nb, int V, double* __restrict__ means) {
    __shared__ double sh[33];
    const double* q = part + (size_t)blockIdx.x * nb;
    double acc = 0.0;
    for (int i = threadIdx.x; i < nb; i += blockDim.x) acc += q[i];
    const double t = block_sum(acc, sh);
    if (threadIdx.x == 0) means[blockIdx.x] = t / (double)V;
}

// Network input: x[r][c] = U_c[r] - <U_c> (c < 2), zero in the padded channels.
__global__ void k_net_in(const float* __restrict__ U, const double* __restrict__ means, int V, int B,
                         bf16* __restrict__ x) {
    const size_t r = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
    if (r >= (size_t)B * V) return;
    const int b = (int)(r / V);
    const size_t i = r - (size_t)b * V;
    const float m0 = (float)means[2 * b], m1 = (float)means[2 * b + 1];
    __align__(16) bf16 v[16];
#pragma unroll
    for (int c = 0; c < 16; ++c) v[c] = __float2bfloat16(0.f);
    v[0] = __float2bfloat16(U[((size_t)2 * b) * V + i] - m0);
    v[1] = __float2bfloat16(U[((size_t)2 * b + 1) * V + i] - m1);
    uint4* dst = (uint4*)(x + r * 16);
    dst[0] = *(const uint4*)&v[0];
    dst[1] = *(const uint4*)&v[8];
}

// Network input with the five x offsets folded into the channels (tcgen05 first layer):
// xf[r][2 dx + c] = U_c[r + dx - 2 along x] - <U_c> for dx = 0..4, zero in channels 10..15, stored
// by channel group within each x row and with two periodic copies on each side of the row,
// [B][nz][ny][2][nx + 4][8] (site x at x + 2), so that a group's part of a tile's staged row,
// x0 - 2 .. x0 + 129, is one contiguous run.
__global__ void k_net_in_fold(const float* __restrict__ U, const double* __restrict__ means, int nx, int V, int B,
                              bf16* __restrict__ xf) {
    const size_t r = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
    if (r >= (size_t)B * V) return;
    const int b = (int)(r / V);
    const int i = (int)(r - (size_t)b * V);
    const int x = i % nx, row = i - x;
    const float m0 = (float)means[2 * b], m1 = (float)means[2 * b + 1];
    const float* U0 = U + ((size_t)2 * b) * V + row;
    const float* U1 = U + ((size_t)2 * b + 1) * V + row;
    __align__(16) bf16 v[16];
#pragma unroll
    for (int dx = 0; dx < 5; ++dx) {
        int xs = x + dx - 2;
        xs = xs < 0 ? xs + nx : (xs >= nx ? xs - nx : xs);
        v[2 * dx] = __float2bfloat16(U0[xs] - m0);
        v[2 * dx + 1] = __float2bfloat16(U1[xs] - m1);
    }
#pragma unroll
    for (int c = 10; c < 16; ++c) v[c] = __float2bfloat16(0.f);
    const size_t rowi = (size_t)b * (V / nx) + row / nx;
    bf16* g0 = xf + rowi * 2 * (size_t)(nx + 4) * 8;   // group 0 of this row; group 1 follows
    bf16* g1 = g0 + (size_t)(nx + 4) * 8;
    const int xp = x + 2;
    *(uint4*)(g0 + (size_t)xp * 8) = *(const uint4*)&v[0];
    *(uint4*)(g1 + (size_t)xp * 8) = *(const uint4*)&v[8];
    const int xh = x < 2 ? x + nx + 2 : (x >= nx - 2 ? x - nx + 2 : -1);   // periodic copy
    if (xh >= 0) {
        *(uint4*)(g0 + (size_t)xh * 8) = *(const uint4*)&v[0];
        *(uint4*)(g1 + (size_t)xh * 8) = *(const uint4*)&v[8];
    }
}

// Channel-last copy h[r][32] of an activation in the padded channel-group layout
// hp[rows][4][nx + 4][8] (site x at x + 2) that the tcgen05 forward writes; for the backward pass.
__global__ void k_unpad32(const bf16* __restrict__ hp, int nx, size_t S, bf16* __restrict__ h) {
    const size_t r = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
    if (r >= S) return;
    const size_t rowi = r / nx;
    const int x = (int)(r - rowi * nx);
    const bf16* src = hp + (rowi * 4 * (size_t)(nx + 4) + (size_t)(x + 2)) * 8;
    uint4* dst = (uint4*)(h + r * 32);
#pragma unroll
    for (int g = 0; g < 4; ++g) dst[g] = *(const uint4*)(src + (size_t)g * (nx + 4) * 8);
}

// Network output: phi_c[r] = phibar_c + y[r][c] - <y_c>  ([B][2][V] float).
__global__ void k_net_out(const float* __restrict__ y, const double* __restrict__ means, int V, int B, double pb0,
                          double pb1, float* __restrict__ phi) {
    const size_t r = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
    if (r >= (size_t)B * V) return;
    const int b = (int)(r / V);
    const size_t i = r - (size_t)b * V;
    const double m0 = means[2 * b], m1 = means[2 * b + 1];
    phi[((size_t)2 * b) * V + i] = (float)(pb0 - m0) + y[r * 16];
    phi[((size_t)2 * b + 1) * V + i] = (float)(pb1 - m1) + y[r * 16 + 1];
}

// Loss gradient: g = (phi - phi*) / n, projected mean-free per sample and channel (the output
// mean removal), written channel-last bf16 [B][V][16]; g is stored first in `gtmp` [B][2][V].
__global__ void k_loss_g(const float* __restrict__ phi, const float* __restrict__ tgt, size_t n, float* __restrict__ g,
                         double* __restrict__ lpart) {
    __shared__ double sh[33];
    float acc = 0.f;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        const float d = phi[i] - tgt[i];
        g[i] = d / (float)n;
        acc += d * d;
    }
    const double t = block_sum((double)acc, sh);
    if (threadIdx.x == 0) lpart[blockIdx.x] = t;
}
__global__ void k_dy(const float* __restrict__ g, const double* __restrict__ means, int V, int B,
                     bf16* __restrict__ dy) {
    const size_t r = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
    if (r >= (size_t)B * V) return;
    const int b = (int)(r / V);
    const size_t i = r - (size_t)b * V;
    const float m0 = (float)means[2 * b], m1 = (float)means[2 * b + 1];
    __align__(16) bf16 v[16];
#pragma unroll
    for (int c = 0; c < 16; ++c) v[c] = __float2bfloat16(0.f);
    v[0] = __float2bfloat16(g[((size_t)2 * b) * V + i] - m0);
    v[1] = __float2bfloat16(g[((size_t)2 * b + 1) * V + i] - m1);
    uint4* dst = (uint4*)(dy + r * 16);
    dst[0] = *(const uint4*)&v[0];
    dst[1] = *(const uint4*)&v[8];
}

// BF16 weights of layer l as mma.sync fragments (the B operand of k_conv): forward Wf with N = output
// and K = input channels (cinp, NT n-tiles of 8), and for the input gradient Wb with N = input and
// K = output channels (coutp, NTb n-tiles) and the offsets reversed; zero in padded channels.  Layout
// [o][lane][k group of 16][n-tile][register][half]: n = 8 j + lane / 4, k = 16 kc + 2 (lane % 4) + 8 r + h.
__global__ void k_prep_w(const float* __restrict__ W, int cin, int cout, int cinp, int coutp, int NT, int NTb,
                         bf16* __restrict__ Wf, bf16* __restrict__ Wb) {
    auto frag = [&](int i, int KC, int nt, int& o, int& n, int& k) {
        const int h = i & 1, r = (i >> 1) & 1;
        int t = i >> 2;
        const int j = t % nt;
        t /= nt;
        const int kc = t % KC;
        t /= KC;
        const int lane = t & 31;
        o = t >> 5;
        n = 8 * j + (lane >> 2);
        k = 16 * kc + 2 * (lane & 3) + 8 * r + h;
    };
    const int step = gridDim.x * blockDim.x, i0 = blockIdx.x * blockDim.x + threadIdx.x;
    int o, n, k;
    for (int i = i0; i < KVOL * NT * 8 * cinp; i += step) {
        frag(i, cinp / 16, NT, o, n, k);
        Wf[i] = __float2bfloat16((n < cout && k < cin) ? W[((size_t)n * cin + k) * KVOL + o] : 0.f);
    }
    if (!Wb) return;
    for (int i = i0; i < KVOL * NTb * 8 * coutp; i += step) {
        frag(i, coutp / 16, NTb, o, n, k);
        Wb[i] = __float2bfloat16((k < cout && n < cin) ? W[((size_t)k * cin + n) * KVOL + (KVOL - 1 - o)] : 0.f);
    }
}

// BF16 weights of a stacked tcgen05 layer: Wt[dz][dx][ci / 8][4 - dy][co][ci % 8] (zero in padded
// channels): per (dz, dx, 8 input channels) the five dy offsets' output channels, last dy first,
// form the rows of one N = 5 CO operand.
__global__ void k_prep_wt_stk(const float* __restrict__ W, int cin, int cout, int cinp, int coutp, bf16* __restrict__ Wt) {
    const int n = KVOL * coutp * cinp;
    const int G = cinp / 8;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        int t = i;
        const int j8 = t % 8;
        t /= 8;
        const int co = t % coutp;
        t /= coutp;
        const int k = t % 5;
        t /= 5;
        const int kc = t % G;
        t /= G;
        const int dx = t % 5, dz = t / 5;
        const int ci = kc * 8 + j8, o = dz * 25 + (4 - k) * 5 + dx;
        const float v = (co < cout && ci < cin) ? W[((size_t)co * cin + ci) * KVOL + o] : 0.f;
        Wt[i] = __float2bfloat16(v);
    }
}

// First-layer weights for the folded input: Wt[dz][dy][k / 8][co][k % 8] with k = 2 dx + ci
// (k < 10), zero for k >= 10.
__global__ void k_prep_wt_fold(const float* __restrict__ W, bf16* __restrict__ Wt) {
    const int n = 25 * 2 * 32 * 8;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const int o2 = i / 512, rem = i % 512;
        const int kc = rem / 256, r2 = rem % 256;
        const int co = r2 / 8, k = kc * 8 + r2 % 8;
        float v = 0.f;
        if (k < 10) v = W[((size_t)co * 2 + (k & 1)) * KVOL + o2 * 5 + (k >> 1)];
        Wt[i] = __float2bfloat16(v);
    }
}

// Adam (FP32 master weights).
__global__ void k_adam(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m, float* __restrict__ v,
                       int n, float lr, float b1, float b2, float eps, float c1, float c2) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const float gi = g[i];
        const float mi = b1 * m[i] + (1.f - b1) * gi;
        const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
        m[i] = mi;
        v[i] = vi;
        p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    }
}

size_t up256(size_t x) { return (x + 255) & ~(size_t)255; }

struct NetLayout {
    size_t params, grads, m, v, wf[NL], wb[NL], wt[NL], x16, x16f, h1, h2, h1p, h2p, y16, dy16, dz2, dz1, gtmp, wpart, part,
        means, lpart, err, bytes;
};
constexpr int kPartBlocks = 512;   // partial sums per channel and sample

// CTAs per dz of a weight gradient: one CTA per SM over the five dz (152 SMs), at most one per tile.
constexpr int kWgradSplits = 30;
int wgrad_splits(int nx, int ny, int nz, int B) {
    const long long t = (long long)B * nz * ((ny + WG_TY - 1) / WG_TY) * (nx / (nx % 32 == 0 ? 32 : 16));
    return t < kWgradSplits ? (int)t : kWgradSplits;
}

NetLayout net_layout(int nx, int ny, int nz, int B) {
    NetLayout L;
    const size_t V = (size_t)nx * ny * nz, S = V * B;
    size_t off = 0;
    auto take = [&](size_t bytes) { const size_t o = off; off = up256(off + bytes); return o; };
    L.params = take(NPARAM * 4);
    L.grads = take(NPARAM * 4);
    L.m = take(NPARAM * 4);
    L.v = take(NPARAM * 4);
    for (int l = 0; l < NL; ++l) {
        L.wf[l] = take((size_t)KVOL * COUTP[l] * CINP[l] * 2);
        L.wb[l] = take((size_t)KVOL * COUTP[l] * CINP[l] * 2);
        L.wt[l] = take((size_t)KVOL * COUTP[l] * CINP[l] * 2);
    }
    L.x16 = take(S * 16 * 2);
    L.x16f = tc_conv_supported(nx, ny) ? take(S / nx * (nx + 4) * 16 * 2) : 0;
    L.h1 = take(S * 32 * 2);
    L.h2 = take(S * 32 * 2);
    // the tcgen05 forward's activations, in the padded channel-group layout [rows][4][nx + 4][8]
    L.h1p = tc_conv_supported(nx, ny) ? take(S / nx * (nx + 4) * 32 * 2) : 0;
    L.h2p = tc_conv_supported(nx, ny) ? take(S / nx * (nx + 4) * 32 * 2) : 0;
    L.y16 = take(S * 16 * 4);
    L.dy16 = take(S * 16 * 2);
    L.dz2 = take(S * 32 * 2);
    L.dz1 = take(S * 32 * 2);
    L.gtmp = take(S * 2 * 4);
    L.wpart = take((size_t)kWgradSplits * KVOL * 32 * 32 * 4);
    const size_t ntc = tc_conv_supported(nx, ny) ? (size_t)tc_conv_blocks(nx, ny, nz) : 0;
    L.part = take((size_t)B * 2 * (ntc > (size_t)kPartBlocks ? ntc : (size_t)kPartBlocks) * 8);
    L.means = take((size_t)B * 2 * 8);
    L.lpart = take((size_t)1024 * 8);
    L.err = take(sizeof(int));
    L.bytes = off;
    return L;
}

size_t poff(int l) {   // offset of layer l's weights in the parameter vector (bias follows)
    size_t o = 0;
    for (int k = 0; k < l; ++k) o += wcount(k) + COUT[k];
    return o;
}

thread_local std::string g_net_err;

}  // namespace

struct dscf_net {
    int nx, ny, nz, B, device;
    size_t V;
    cudaStream_t stream;
    char* ws;
    NetLayout L;
    int adam_t = 0;
    int path = 0;          // 0: tcgen05 forward where the grid allows it, 1: mma.sync only
    bool tc_ok = false;    // grid and device allow the tcgen05 forward
    std::string err;
    bool use_tc() const { return tc_ok && path == 0; }
    template <typename P> P* at(size_t off) { return (P*)(ws + off); }
};

namespace {

int nfail(dscf_net* n, int code, const char* msg) {
    if (n) n->err = msg; else g_net_err = msg;
    return code;
}
int ncheck(dscf_net* n, cudaError_t e, const char* what) {
    if (e == cudaSuccess) return DSCF_OK;
    std::string m = std::string(what) + ": " + cudaGetErrorString(e);
    return nfail(n, DSCF_ERR_CUDA, m.c_str());
}

void prep_weights(dscf_net* n) {
    for (int l = 0; l < NL; ++l)
        k_prep_w<<<128, 256, 0, n->stream>>>(n->at<float>(n->L.params) + poff(l), CIN[l], COUT[l], CINP[l], COUTP[l],
                                               NTF[l], CINP[l] / 8, n->at<bf16>(n->L.wf[l]),
                                               l > 0 ? n->at<bf16>(n->L.wb[l]) : nullptr);
    if (n->tc_ok) {
        k_prep_wt_fold<<<64, 256, 0, n->stream>>>(n->at<float>(n->L.params) + poff(0), n->at<bf16>(n->L.wt[0]));
        for (int l = 1; l < NL; ++l)
            k_prep_wt_stk<<<64, 256, 0, n->stream>>>(n->at<float>(n->L.params) + poff(l), CIN[l], COUT[l], CINP[l],
                                                       COUTP[l], n->at<bf16>(n->L.wt[l]));
    }
}

// Blocks of a channel sum: up to kPartBlocks x 256 sites every thread would have at most one site, so
// the wide form takes 16 per thread instead.
bool chan_wide(const dscf_net* n) { return n->V <= (size_t)kPartBlocks * 256; }
int chan_blocks(const dscf_net* n) { return chan_wide(n) ? (int)((n->V + 4095) / 4096) : kPartBlocks; }
// means of C = 2 channels of a [B][C][V] field into L.means
void chan_means(dscf_net* n, const float* f, int C) {
    const int nb = chan_blocks(n);
    const dim3 grid(nb, C, n->B);
    if (chan_wide(n)) k_chan_parts<true><<<grid, 256, 0, n->stream>>>(f, C, (int)n->V, n->at<double>(n->L.part));
    else k_chan_parts<false><<<grid, 256, 0, n->stream>>>(f, C, (int)n->V, n->at<double>(n->L.part));
    k_chan_final<<<C * n->B, 256, 0, n->stream>>>(n->at<double>(n->L.part), nb, (int)n->V, n->at<double>(n->L.means));
}

// mma.sync convolution and weight gradient of the network's grid
template <int CI, int NT, int EPI, int MX>
void conv_mx(dscf_net* n, const bf16* in, const bf16* W, const float* bias, int cout, const bf16* hact, void* out, float* bgrad) {
    using CT = ConvTile<MX>;
    constexpr int smem = CT::SITES * CI * 2;
    const int blocks = n->B * (n->nx / (16 * MX)) * ((n->ny + CV_TY - 1) / CV_TY) * ((n->nz + CT::TZ - 1) / CT::TZ);
    k_conv<CI, NT, EPI, MX><<<blocks, 128, smem, n->stream>>>(in, (const uint4*)W, bias, cout, hact, out, n->nx, n->ny, n->nz, bgrad);
}
template <int CI, int NT, int EPI>
void conv(dscf_net* n, const bf16* in, const bf16* W, const float* bias, int cout, const bf16* hact, void* out, float* bgrad) {
    if (n->nx % 32 == 0) conv_mx<CI, NT, EPI, 2>(n, in, W, bias, cout, hact, out, bgrad);
    else conv_mx<CI, NT, EPI, 1>(n, in, W, bias, cout, hact, out, bgrad);
}
template <int CI, int NT, int CD, int MX>
void wgrad_mx(dscf_net* n, const bf16* in, const bf16* dout, int nsplit) {
    using WT = WgTile<CI, NT, CD, MX>;
    constexpr int smem = WT::SMEM;
    k_wgrad<CI, NT, CD, MX><<<dim3(nsplit, 5), 32 * WG_WARPS, smem, n->stream>>>(in, dout, n->at<float>(n->L.wpart), n->nx, n->ny, n->nz, n->B);
}
template <int CI, int NT, int CD>
void wgrad(dscf_net* n, int l, const bf16* in, const bf16* dout, float* dW) {
    const int nsplit = wgrad_splits(n->nx, n->ny, n->nz, n->B);
    if (n->nx % 32 == 0) wgrad_mx<CI, NT, CD, 2>(n, in, dout, nsplit);
    else wgrad_mx<CI, NT, CD, 1>(n, in, dout, nsplit);
    k_wgrad_sum<<<(KVOL * CI * 8 * NT + 255) / 256, 256, 0, n->stream>>>(n->at<float>(n->L.wpart), nsplit, CI, 8 * NT, CIN[l], COUT[l], dW);
}

// Dynamic shared memory of the kernels above, once per network (cudaError_t of the first failure).
template <int CI, int NT, int EPI, int MX>
cudaError_t conv_smem() {
    return cudaFuncSetAttribute(k_conv<CI, NT, EPI, MX>, cudaFuncAttributeMaxDynamicSharedMemorySize, ConvTile<MX>::SITES * CI * 2);
}
template <int CI, int NT, int CD, int MX>
cudaError_t wgrad_smem() {
    using WT = WgTile<CI, NT, CD, MX>;
    return cudaFuncSetAttribute(k_wgrad<CI, NT, CD, MX>, cudaFuncAttributeMaxDynamicSharedMemorySize, WT::SMEM);
}
template <int MX>
cudaError_t mma_prepare() {
    cudaError_t e = conv_smem<16, 4, EPI_TANH, MX>();
    if (e == cudaSuccess) e = conv_smem<32, 4, EPI_TANH, MX>();
    if (e == cudaSuccess) e = conv_smem<32, 1, EPI_LIN_F32, MX>();
    if (e == cudaSuccess) e = conv_smem<16, 4, EPI_DTANH, MX>();
    if (e == cudaSuccess) e = conv_smem<32, 4, EPI_DTANH, MX>();
    if (e == cudaSuccess) e = wgrad_smem<32, 1, 16, MX>();
    if (e == cudaSuccess) e = wgrad_smem<32, 4, 32, MX>();
    if (e == cudaSuccess) e = wgrad_smem<16, 4, 32, MX>();
    return e;
}

// forward pass from U ([B][2][V] float, device) to phi ([B][2][V] float, device)
void forward(dscf_net* n, const float* U, double pb0, double pb1, float* phi) {
    const int V = (int)n->V, B = n->B;
    const int eb = (int)((n->V * B + 255) / 256);
    chan_means(n, U, 2);
    k_net_in<<<eb, 256, 0, n->stream>>>(U, n->at<double>(n->L.means), V, B, n->at<bf16>(n->L.x16));
    if (n->use_tc()) {
        k_net_in_fold<<<eb, 256, 0, n->stream>>>(U, n->at<double>(n->L.means), n->nx, V, B, n->at<bf16>(n->L.x16f));
        const size_t act[NL + 1] = {n->L.x16f, n->L.h1p, n->L.h2p, n->L.y16};
        for (int l = 0; l < NL; ++l)
            launch_conv_tc(l, n->ws + act[l], n->ws + n->L.wt[l], n->at<float>(n->L.params) + poff(l) + wcount(l),
                           COUT[l], n->ws + act[l + 1], n->nx, n->ny, n->nz, B, n->at<double>(n->L.part),
                           n->at<int>(n->L.err), n->stream);
        // the output layer left per-CTA sums of its two channels
        k_chan_final<<<2 * B, 256, 0, n->stream>>>(n->at<double>(n->L.part), tc_conv_blocks(n->nx, n->ny, n->nz), V,
                                                   n->at<double>(n->L.means));
    } else {
        const float* prm = n->at<float>(n->L.params);
        conv<16, 4, EPI_TANH>(n, n->at<bf16>(n->L.x16), n->at<bf16>(n->L.wf[0]), prm + poff(0) + wcount(0), 32, nullptr,
                              n->at<bf16>(n->L.h1), nullptr);
        conv<32, 4, EPI_TANH>(n, n->at<bf16>(n->L.h1), n->at<bf16>(n->L.wf[1]), prm + poff(1) + wcount(1), 32, nullptr,
                              n->at<bf16>(n->L.h2), nullptr);
        conv<32, 1, EPI_LIN_F32>(n, n->at<bf16>(n->L.h2), n->at<bf16>(n->L.wf[2]), prm + poff(2) + wcount(2), 2, nullptr,
                                 n->at<float>(n->L.y16), nullptr);
        const int nb = chan_blocks(n);
        const dim3 grid(nb, 2, B);
        if (chan_wide(n)) k_chan_parts_cl<true><<<grid, 256, 0, n->stream>>>(n->at<float>(n->L.y16), 2, 16, V, n->at<double>(n->L.part));
        else k_chan_parts_cl<false><<<grid, 256, 0, n->stream>>>(n->at<float>(n->L.y16), 2, 16, V, n->at<double>(n->L.part));
        k_chan_final<<<2 * B, 256, 0, n->stream>>>(n->at<double>(n->L.part), nb, V, n->at<double>(n->L.means));
    }
    k_net_out<<<eb, 256, 0, n->stream>>>(n->at<float>(n->L.y16), n->at<double>(n->L.means), V, B, pb0, pb1, phi);
}

// gradient of 0.5 mean((phi - target)^2) with respect to all parameters, into grads
void backward(dscf_net* n, const float* phi, const float* tgt) {
    const int V = (int)n->V, B = n->B;
    const size_t S = n->V * B;
    const int eb = (int)((S + 255) / 256);
    float* grads = n->at<float>(n->L.grads);
    if (n->use_tc()) {   // the forward pass left its activations in the padded layout
        k_unpad32<<<eb, 256, 0, n->stream>>>(n->at<bf16>(n->L.h1p), n->nx, S, n->at<bf16>(n->L.h1));
        k_unpad32<<<eb, 256, 0, n->stream>>>(n->at<bf16>(n->L.h2p), n->nx, S, n->at<bf16>(n->L.h2));
    }
    cudaMemsetAsync(grads, 0, NPARAM * 4, n->stream);
    k_loss_g<<<1024, 256, 0, n->stream>>>(phi, tgt, S * 2, n->at<float>(n->L.gtmp), n->at<double>(n->L.lpart));
    chan_means(n, n->at<float>(n->L.gtmp), 2);
    k_dy<<<eb, 256, 0, n->stream>>>(n->at<float>(n->L.gtmp), n->at<double>(n->L.means), V, B, n->at<bf16>(n->L.dy16));
    // layer 3
    wgrad<32, 1, 16>(n, 2, n->at<bf16>(n->L.h2), n->at<bf16>(n->L.dy16), grads + poff(2));
    // the output bias cannot change phi_hat (its per-sample mean is removed): its gradient is zero
    conv<16, 4, EPI_DTANH>(n, n->at<bf16>(n->L.dy16), n->at<bf16>(n->L.wb[2]), nullptr, 32, n->at<bf16>(n->L.h2),
                           n->at<bf16>(n->L.dz2), grads + poff(1) + wcount(1));
    // layer 2
    wgrad<32, 4, 32>(n, 1, n->at<bf16>(n->L.h1), n->at<bf16>(n->L.dz2), grads + poff(1));
    conv<32, 4, EPI_DTANH>(n, n->at<bf16>(n->L.dz2), n->at<bf16>(n->L.wb[1]), nullptr, 32, n->at<bf16>(n->L.h1),
                           n->at<bf16>(n->L.dz1), grads + poff(0) + wcount(0));
    // layer 1
    wgrad<16, 4, 32>(n, 0, n->at<bf16>(n->L.x16), n->at<bf16>(n->L.dz1), grads + poff(0));
}

// splitmix64-based normal deviates for the initial weights (Box-Muller)
double u01(uint64_t seed, uint64_t k) {
    uint64_t z = seed + (k + 1) * 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    z ^= z >> 31;
    return (double)(z >> 11) * (1.0 / 9007199254740992.0);
}

}  // namespace

bool dscf_net_fits(const dscf_net* n, int nx, int ny, int nz) {
    return n && n->nx == nx && n->ny == ny && n->nz == nz && n->B == 1;
}
int dscf_net_forward_launches(const dscf_net* n) { return 9; }
void dscf_net_forward_on(dscf_net* n, cudaStream_t stream, const float* U, double pb0, double pb1, float* phi) {
    cudaStream_t keep = n->stream;
    n->stream = stream;
    forward(n, U, pb0, pb1, phi);
    n->stream = keep;
}

extern "C" {

size_t dscf_net_workspace_bytes(int32_t nx, int32_t ny, int32_t nz, int32_t batch) {
    if (nx < 16 || nx % 16 || ny < 1 || nz < 1 || batch < 1) return 0;
    return net_layout(nx, ny, nz, batch).bytes;
}

int dscf_net_init(int32_t nx, int32_t ny, int32_t nz, int32_t batch, uint64_t seed, void* workspace, size_t bytes,
                  void* stream, dscf_net** out) {
    if (!out) return nfail(nullptr, DSCF_ERR_ARG, "out is NULL");
    *out = nullptr;
    const size_t need = dscf_net_workspace_bytes(nx, ny, nz, batch);
    if (need == 0) return nfail(nullptr, DSCF_ERR_ARG, "need nx a multiple of 16, ny, nz, batch >= 1");
    if (!workspace || ((uintptr_t)workspace & 255)) return nfail(nullptr, DSCF_ERR_ARG, "workspace must be 256-byte aligned");
    if (bytes < need) return nfail(nullptr, DSCF_ERR_OOM, "workspace too small");
    cudaPointerAttributes pa;
    if (cudaPointerGetAttributes(&pa, workspace) != cudaSuccess || pa.type != cudaMemoryTypeDevice) {
        cudaGetLastError();
        return nfail(nullptr, DSCF_ERR_ARG, "workspace is not device memory");
    }
    dscf_net* n = new (std::nothrow) dscf_net;
    if (!n) return nfail(nullptr, DSCF_ERR_OOM, "host allocation failed");
    n->nx = nx; n->ny = ny; n->nz = nz; n->B = batch; n->device = pa.device;
    n->V = (size_t)nx * ny * nz;
    n->stream = (cudaStream_t)stream;
    n->ws = (char*)workspace;
    n->L = net_layout(nx, ny, nz, batch);
    cudaSetDevice(n->device);
    {
        int major = 0, minor = 0;
        cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, n->device);
        cudaDeviceGetAttribute(&minor, cudaDevAttrComputeCapabilityMinor, n->device);
        n->tc_ok = tc_conv_supported(nx, ny) && major == 10 && minor == 3 && tc_conv_prepare() == 0;
        cudaGetLastError();
    }
    // Glorot-like normal initial weights, zero biases
    std::vector<float> p(NPARAM, 0.f);
    uint64_t k = 0;
    for (int l = 0; l < NL; ++l) {
        const double sd = std::sqrt(2.0 / ((double)(CIN[l] + COUT[l]) * KVOL));
        float* w = p.data() + poff(l);
        for (size_t i = 0; i < wcount(l); ++i, k += 2) {
            const double u1 = 1.0 - u01(seed, k), u2 = u01(seed, k + 1);
            w[i] = (float)(sd * std::sqrt(-2.0 * std::log(u1)) * std::cos(6.283185307179586 * u2));
        }
    }
    int rc = ncheck(n, nx % 32 == 0 ? mma_prepare<2>() : mma_prepare<1>(), "shared-memory limit");
    if (!rc) rc = ncheck(n, cudaMemcpy(n->at<float>(n->L.params), p.data(), NPARAM * 4, cudaMemcpyHostToDevice), "params");
    if (!rc) rc = ncheck(n, cudaMemset(n->at<float>(n->L.m), 0, NPARAM * 4), "m");
    if (!rc) rc = ncheck(n, cudaMemset(n->at<float>(n->L.v), 0, NPARAM * 4), "v");
    if (!rc) rc = ncheck(n, cudaMemset(n->at<int>(n->L.err), 0, sizeof(int)), "error word");
    if (!rc) {
        prep_weights(n);
        rc = ncheck(n, cudaStreamSynchronize(n->stream), "init");
    }
    if (rc) { g_net_err = n->err; delete n; return rc; }
    *out = n;
    return DSCF_OK;
}

int dscf_net_forward(dscf_net* n, const float* U, const double* phibar, float* phi_out) {
    if (!n || !U || !phibar || !phi_out) return n ? nfail(n, DSCF_ERR_ARG, "NULL argument") : DSCF_ERR_ARG;
    cudaSetDevice(n->device);
    forward(n, U, phibar[0], phibar[1], phi_out);
    return ncheck(n, cudaGetLastError(), "net forward");
}

int dscf_net_gradient(dscf_net* n, const float* U, const float* phi_target, const double* phibar, float* phi_work,
                      double* loss, float* grads_out) {
    if (!n || !U || !phi_target || !phibar || !phi_work) return n ? nfail(n, DSCF_ERR_ARG, "NULL argument") : DSCF_ERR_ARG;
    cudaSetDevice(n->device);
    forward(n, U, phibar[0], phibar[1], phi_work);
    backward(n, phi_work, phi_target);
    int rc = ncheck(n, cudaGetLastError(), "net gradient");
    if (rc) return rc;
    if (loss) {
        std::vector<double> lp(1024);
        rc = ncheck(n, cudaMemcpyAsync(lp.data(), n->at<double>(n->L.lpart), 1024 * 8, cudaMemcpyDeviceToHost, n->stream),
                    "loss");
        if (!rc) rc = ncheck(n, cudaStreamSynchronize(n->stream), "loss sync");
        if (rc) return rc;
        double s = 0.0;
        for (double v : lp) s += v;
        *loss = 0.5 * s / (double)(n->V * n->B * 2);
    }
    if (grads_out)
        return ncheck(n, cudaMemcpyAsync(grads_out, n->at<float>(n->L.grads), NPARAM * 4, cudaMemcpyDeviceToDevice, n->stream),
                      "grads");
    return DSCF_OK;
}

int dscf_net_train_step(dscf_net* n, const float* U, const float* phi_target, const double* phibar, float* phi_work,
                        float lr, double* loss) {
    int rc = dscf_net_gradient(n, U, phi_target, phibar, phi_work, loss, nullptr);
    if (rc) return rc;
    n->adam_t += 1;
    const float b1 = 0.9f, b2 = 0.999f;
    const float c1 = 1.f - std::pow(b1, (float)n->adam_t), c2 = 1.f - std::pow(b2, (float)n->adam_t);
    k_adam<<<256, 256, 0, n->stream>>>(n->at<float>(n->L.params), n->at<float>(n->L.grads), n->at<float>(n->L.m),
                                       n->at<float>(n->L.v), (int)NPARAM, lr, b1, b2, 1e-8f, c1, c2);
    prep_weights(n);
    return ncheck(n, cudaGetLastError(), "adam");
}

int dscf_net_get_params(dscf_net* n, float* dst) {
    if (!n || !dst) return DSCF_ERR_ARG;
    return ncheck(n, cudaMemcpyAsync(dst, n->at<float>(n->L.params), NPARAM * 4, cudaMemcpyDefault, n->stream), "get params");
}

int dscf_net_set_params(dscf_net* n, const float* src) {
    if (!n || !src) return DSCF_ERR_ARG;
    int rc = ncheck(n, cudaMemcpyAsync(n->at<float>(n->L.params), src, NPARAM * 4, cudaMemcpyDefault, n->stream), "set params");
    if (rc) return rc;
    prep_weights(n);
    n->adam_t = 0;
    cudaMemsetAsync(n->at<float>(n->L.m), 0, NPARAM * 4, n->stream);
    cudaMemsetAsync(n->at<float>(n->L.v), 0, NPARAM * 4, n->stream);
    return ncheck(n, cudaGetLastError(), "set params");
}

int64_t dscf_net_num_params(void) { return (int64_t)NPARAM; }

int dscf_net_set_tensor_path(dscf_net* n, int32_t path) {
    if (!n) return DSCF_ERR_ARG;
    if (path != 0 && path != 1) return nfail(n, DSCF_ERR_ARG, "path must be 0 (tcgen05 where possible) or 1 (mma.sync)");
    cudaSetDevice(n->device);
    int rc = ncheck(n, cudaStreamSynchronize(n->stream), "path sync");
    if (rc) return rc;
    n->path = path;
    return DSCF_OK;
}

int32_t dscf_net_tensor_path(const dscf_net* n) { return n ? (n->use_tc() ? 2 : 1) : 0; }

int dscf_net_status(dscf_net* n) {
    if (!n) return DSCF_ERR_ARG;
    cudaSetDevice(n->device);
    int e = 0;
    int rc = ncheck(n, cudaStreamSynchronize(n->stream), "status sync");
    if (!rc) rc = ncheck(n, cudaMemcpy(&e, n->at<int>(n->L.err), sizeof(int), cudaMemcpyDeviceToHost), "status read");
    if (rc) return rc;
    if (e) {
        cudaMemset(n->at<int>(n->L.err), 0, sizeof(int));
        return nfail(n, DSCF_ERR_TIMEOUT, "a tensor-core convolution gave up waiting for its MMAs");
    }
    return DSCF_OK;
}

int dscf_net_free(dscf_net* n) {
    delete n;
    return DSCF_OK;
}

const char* dscf_net_last_error(const dscf_net* n) { return n ? n->err.c_str() : g_net_err.c_str(); }

}  // extern "C"
