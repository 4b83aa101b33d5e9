// Boltzmann factors of the density evaluations.  (The contour sweeps are in dscf_coop.cuh, any grid, and
// dscf_pers.cu, bricks.)
#include "dscf_internal.cuh"

#include <cstdint>
#include <type_traits>

namespace dscf {

// Boltzmann factors E_I = exp(-U'_I) for the potential U' of the next gradient evaluation:
//   mode 0: U' = U;  mode 1 (trial): U' = U + a1 d with a1 = -<g,d>/<d,phi_m d>;
//   mode 2 (commit): secant step a = a1 (-h0)/(h1 - h0), U <- U + a d, U' = U;
//   mode 3: U' = external potential (forward density map alone).
// The copolymer's factors carry a weight against the growth of the sweeps' passes, which leave out their
// centre weights (Par::ew).  Also the FP64 partial sums of exp(-U'_S) for the solvent
// normalisation.
template <typename T>
__global__ void __launch_bounds__(kFlatThreads) k_exp(const Rep* __restrict__ reps, const int* __restrict__ blk2rep,
                                                      int mode, int k, const T* __restrict__ Uext, int write_u) {
    __shared__ double sh[3 * 33];
    const Rep& R = reps[blk2rep[blockIdx.x]];
    const int lb = blockIdx.x - R.blk0;
    const long long V = R.V;
    const long long i0 = (long long)lb * R.chunk;
    const long long i1 = min(i0 + (long long)R.chunk, V);
    __shared__ T ta_sh;
    if (threadIdx.x == 0) {   // the step length, once per block (FP64 divisions)
        double a = 0.0;
        if (mode == 1 || mode == 2) {
            // totals of the direction and trial kernels' partials, formed by their last blocks
            const double h0 = R.scal[S_H0S], cd = R.scal[S_CDS];
            const double q = h0 / cd;
            const double a1 = (cd > 0.0 && isfinite(q)) ? -q : 0.0;
            a = a1;
            if (mode == 2) {
                const double den = R.scal[S_H1S] - h0;
                a = (den > 0.0) ? a1 * (-h0) / den : a1;
                // With the learned predictor the secant is capped at the local-curvature step a1: the
                // exact response is stiffer than the local one (a <= a1), and a network whose response
                // to the tiny trial displacement is below its resolution would otherwise give a
                // near-zero secant denominator and an unbounded step.
                if (write_u && a > a1) a = a1;
                if (lb == 0) {
                    R.scal[S_ITER0 + 4 * k + 0] = a1;
                    R.scal[S_ITER0 + 4 * k + 1] = a;
                }
            }
        }
        ta_sh = (T)a;
    }
    if (mode == 1 && k == 0 && lb == 0) {
        // start-of-inversion residual (partials written by the direction kernel)
        const double gg = reduce_parts(slot(R, P_GG0), R.nblk, sh);
        const double gm = reduce_parts_max(slot(R, P_GMAX), R.nblk, sh);
        if (threadIdx.x == 0) {
            R.scal[S_GG0] = gg;
            R.scal[S_GMAX0] = gm;
        }
    }
    __syncthreads();
    const int ns = R.ns;
    // distinct fields: no store below can change a value loaded from another of them
    T* __restrict__ U = (T*)R.U;
    const T* __restrict__ d = (const T*)R.d;
    T* __restrict__ E = (T*)R.E;
    const T ta = ta_sh, ew = pars<T>(R).ew;
    double es = 0.0;   // sum of exp(-U_S) of the scalar loop
    float es4 = 0.f;   // and of the vector loop
    bool vec = false;
    // (the caller's field may begin at any element: 16-byte accesses only where its blocks are aligned)
    if constexpr (sizeof(T) == 4) vec = (V & 3) == 0 && (mode != 3 || ((uintptr_t)(Uext + R.ext_off) & 15) == 0);
    if (vec) {   // FP32, 4 consecutive sites per thread and iteration (16-byte accesses)
        const float fa = (float)ta;
        const int j0 = (int)i0, j1 = (int)i1;
        constexpr int S = 4 * kFlatThreads;   // sites per block-wide iteration
        // UB iterations of NS species at a time: every load of the batch is issued before the
        // first use (a thread has only a few iterations, so a plain loop would wait for each)
        auto run = [&](auto nsc, auto ubc) {
            constexpr int NS = decltype(nsc)::value, UB = decltype(ubc)::value;
            for (int ib = j0 + 4 * (int)threadIdx.x; ib < j1; ib += UB * S) {
                float4 uu[UB][NS], dv[UB][NS];
#pragma unroll
                for (int it = 0; it < UB; ++it)
#pragma unroll
                    for (int I = 0; I < NS; ++I) {
                        const int i = ib + it * S;
                        if (i < j1) {
                            const size_t o = (size_t)I * V + i;
                            uu[it][I] = (mode == 3) ? *(const float4*)((const float*)Uext + R.ext_off + o)
                                                    : *(const float4*)((const float*)U + o);
                            if (mode == 1 || mode == 2) dv[it][I] = *(const float4*)((const float*)d + o);
                        }
                    }
#pragma unroll
                for (int it = 0; it < UB; ++it)
#pragma unroll
                    for (int I = 0; I < NS; ++I) {
                        const int i = ib + it * S;
                        if (i < j1) {
                            const size_t o = (size_t)I * V + i;
                            float4 u = uu[it][I];
                            if (mode == 1 || mode == 2) {
                                const float4 dd = dv[it][I];
                                u.x += fa * dd.x;
                                u.y += fa * dd.y;
                                u.z += fa * dd.z;
                                u.w += fa * dd.w;
                                if (mode == 2) *(float4*)((float*)U + o) = u;
                            }
                            const float w = I == 2 ? 1.f : (float)ew;   // the solvent has no stencil
                            const float4 e =
                                write_u ? u : make_float4(w * bexp(u.x), w * bexp(u.y), w * bexp(u.z), w * bexp(u.w));
                            *(float4*)((float*)E + o) = e;
                            if (I == 2) es4 += (e.x + e.y) + (e.z + e.w);
                        }
                    }
            }
        };
        if (ns == 2) run(std::integral_constant<int, 2>{}, std::integral_constant<int, 2>{});
        else run(std::integral_constant<int, 3>{}, std::integral_constant<int, 1>{});
    }
    for (int I = 0; I < ns && !vec; ++I) {
        for (long long i = i0 + threadIdx.x; i < i1; i += kFlatThreads) {
            const long long o = (long long)I * V + i;
            T u;
            if (mode == 0) {
                u = U[o];
            } else if (mode == 1) {
                u = U[o] + ta * d[o];
            } else if (mode == 2) {
                u = U[o] + ta * d[o];
                U[o] = u;
            } else {
                u = Uext[R.ext_off + o];
            }
            const T e = write_u ? u : (I == 2 ? bexp(u) : ew * bexp(u));   // write_u: the learned predictor takes U' itself
            E[o] = e;
            if (I == 2) es += (double)e;
        }
    }
    if (ns == 3) {
        double t[1] = {es};
        if (vec) {
            const float v[1] = {es4};
            block_total<1>(v, sh, t);
        } else {
            block_sum_n<1>(t, sh);
        }
        if (threadIdx.x == 0) slot(R, P_ES)[lb] = t[0];
        __shared__ int fin;
        if (R.nq == 0 && last_block_of(R, &fin)) {   // (nq: the allocation-free path sums in norm_of)
            if constexpr (sizeof(T) == 8) {
                if (threadIdx.x < 32) {
                    const Two s = total_of(slot(R, P_ES), R.nblk);
                    if (threadIdx.x == 0) {
                        R.scal[S_ESS] = s.hi;
                        R.scal[S_ESLO] = s.lo;
                    }
                }
            } else {
                const double s = reduce_parts_cg(slot(R, P_ES), R.nblk, sh);
                if (threadIdx.x == 0) R.scal[S_ESS] = s;
            }
        }
    }
}

template <typename T>
void launch_exp(const Launch& L, int mode, int k, const void* Uext, int write_u) {
    k_exp<T><<<L.nblk_total, kFlatThreads, 0, L.stream>>>(L.reps, L.blk2rep, mode, k, (const T*)Uext, write_u);
}

template void launch_exp<double>(const Launch&, int, int, const void*, int);
template void launch_exp<float>(const Launch&, int, int, const void*, int);

}  // namespace dscf
