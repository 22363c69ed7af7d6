// kern_forward64.cu -- the forward problem (FP of Sec. 2.2) in FP64: reference
// traces and misfits, every state update compensated, in the affine form of
// the RK4 step (afm_affine.cuh).
//
// What bounds it is the issue of FP64 instructions: an SM sub-partition takes
// one warp's FP64 instruction every 64 clocks however many of its lanes are
// active, so a step costs 64 clocks times its FP64 instruction count.
//   many candidates   one thread each (fwd64_kernel), ~170 FP64 instructions
//                     per step for three modes and the DMT law (~240 with the
//                     stages evaluated mode by mode and a reciprocal and a
//                     square root in every force)
//   few (one warp per sub-partition at most)   L lanes per candidate, one
//                     mode each, and for rate-free laws the stage forces
//                     split between even lanes (F1, F3) and odd lanes (F2,
//                     F4): ~80 FP64 instructions per step; the shuffles
//                     between the lanes cost two 32-bit instructions each
#include <type_traits>

#include "afm_affine.cuh"
#include "afm_device.cuh"
#include "afm_launch.h"

namespace afm {

namespace {

template <typename F>
cudaError_t dispatch_mf(int m, int force, F&& f) {
    auto byF = [&](auto Mc) -> cudaError_t {
        switch (force) {
            case F_LINEAR: return f(Mc, std::integral_constant<int, F_LINEAR>{});
            case F_DMT: return f(Mc, std::integral_constant<int, F_DMT>{});
            case F_DMT_KV: return f(Mc, std::integral_constant<int, F_DMT_KV>{});
            case F_HOOKE: return f(Mc, std::integral_constant<int, F_HOOKE>{});
            case F_SPRING_DAMPER: return f(Mc, std::integral_constant<int, F_SPRING_DAMPER>{});
        }
        return cudaErrorInvalidValue;
    };
    if (m == 1) return byF(std::integral_constant<int, 1>{});
    if (m == 3) return byF(std::integral_constant<int, 3>{});
    return byF(std::integral_constant<int, AFM_MAXM>{});
}

__device__ __forceinline__ void store_misfit64(double s, double* S, int p, int* flags) {
    if (!(s < (double)INFINITY)) {
        s = (double)INFINITY;
        if (flags != nullptr) atomicAdd(flags, 1);
    }
    S[p] = s;
}

}  // namespace

template <int M, int FORCE>
__global__ void __launch_bounds__(128)
fwd64_kernel(const KAffine<double> K, const double* __restrict__ x, int P,
             double* __restrict__ defl, const double* __restrict__ U, double* __restrict__ S,
             int* __restrict__ flags) {
    extern __shared__ __align__(16) double tab[];
    aff::build_rows<double, M, FORCE>(K, tab);
    __syncthreads();
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= P) return;
    double xd[AFM_MAXD];
    for (int d = 0; d < K.D; ++d) xd[d] = x[(size_t)d * P + p];
    const aff::LawCoef<double> c = aff::law_coef(make_coef<double, double>(K, xd));
    constexpr int W = aff::Rows<M, FORCE>::words, WS = aff::Table<double, M, FORCE>::stride;
    aff::State<double, M, aff::ALL> s;
    aff::init<double, M, aff::ALL>(K, s);
    double Sm = 0.0, cS = 0.0;
    const double* row = tab;
    const double* end = tab + (size_t)(K.spc2 >> 1) * WS;
    for (int k = 0; k < K.n_steps; ++k) {
        double R[W];
        aff::load_row<double, M, FORCE>(K, row, R);
        row += WS;
        if (row == end) row = tab;
        aff::step<double, M, FORCE, aff::ALL>(K, c, R, s);
        const double u = aff::tip(s);
        if (defl != nullptr) defl[(size_t)k * P + p] = u;
        if (U != nullptr) aff::misfit_add(U[k], u, Sm, cS);
    }
    if (S != nullptr) store_misfit64(Sm, S, p, flags);
}

// Lanes per candidate: one mode each, and at least two for the stage split.
template <int M>
struct Lanes64 {
    static constexpr int value = M == 1 ? 2 : M <= 4 ? 4 : 8;
};

template <int L>
__device__ __forceinline__ double group_sum64(double v) {
#pragma unroll
    for (int o = 1; o < L; o <<= 1) v = aff::add(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

// Sums of a over the group on its even lanes and of b on its odd lanes: the
// first exchange hands each lane the neighbour's part of its own sum.
template <int L>
__device__ __forceinline__ double group_sum64_split(double a, double b, bool odd) {
    const double other = __shfl_xor_sync(0xffffffffu, odd ? a : b, 1);
    double v = aff::add(odd ? b : a, other);
#pragma unroll
    for (int o = 2; o < L; o <<= 1) v = aff::add(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

template <int M, int FORCE>
__global__ void __launch_bounds__(128, 1)
fwd64_lanes_kernel(const KAffine<double> K, const double* __restrict__ x, int P, int wpb,
                   double* __restrict__ defl, const double* __restrict__ U,
                   double* __restrict__ S, int* __restrict__ flags) {
    constexpr int L = Lanes64<M>::value, G = 32 / L;
    constexpr bool rate = UsesRate<FORCE>::value;
    extern __shared__ __align__(16) double tab[];
    aff::build_rows<double, M, FORCE>(K, tab);
    __syncthreads();
    const int warp = threadIdx.x >> 5, wl = threadIdx.x & 31;
    if (warp >= wpb) return;
    const int first = (blockIdx.x * wpb + warp) * G;
    if (first >= P) return;   // whole warps
    const int p0 = first + wl / L, ln = wl % L;
    const int p = min(p0, P - 1);
    const bool owner = p0 < P && ln == 0, odd = (ln & 1) != 0;
    double xd[AFM_MAXD];
    for (int d = 0; d < K.D; ++d) xd[d] = x[(size_t)d * P + p];
    const aff::LawCoef<double> c = aff::law_coef(make_coef<double, double>(K, xd));
    // this lane's mode: 0 past the last one, with every constant zero
    const Affine<double>& A = K.af;
    const bool real = ln < M;
    const int i = real ? ln : 0;
    const double on = real ? 1.0 : 0.0;
    const bool m0 = i == 0;
    // stage gaps as full forms (q_0's own term included), increments
    const double g2q = on * (m0 ? 1.0 + A.d2q : 1.0), g2p = on * (m0 ? A.d2w : 1.0);
    const double g3q = on * (m0 ? 1.0 + A.d3q[0] : A.d3q[i]), g3p = on * A.d3p[i];
    const double g4q = on * (m0 ? 1.0 + A.d4q[0] : A.d4q[i]), g4p = on * A.d4p[i];
    const double A1 = m0 ? 0.0 : A.A1[i], B = on * (m0 ? 1.0 : A.B[i]);
    const double Cq = on * (m0 ? A.c0 : A.C[i]), D1 = on * (m0 ? A.c0 + A.ec : A.D1[i]);
    double bq[3], bp[4];
#pragma unroll
    for (int k = 0; k < 3; ++k) bq[k] = on * A.bq[k][i];
#pragma unroll
    for (int k = 0; k < 4; ++k) bp[k] = on * A.bp[k][i];
    double r1q = 0, r1p = 0, r2q = 0, r2p = 0, r3q = 0, r3p = 0, r4q = 0, r4p = 0;
    if constexpr (rate) {
        r1q = on * (m0 ? A.v1q : 0.0);
        r1p = on * (m0 ? A.v1w : A.third);
        r2q = on * A.r2q[i];
        r2p = on * A.r2p[i];
        r3q = on * A.r3q[i];
        r3p = on * A.r3p[i];
        r4q = on * A.r4q[i];
        r4p = on * A.r4p[i];
    }
    const double ea = odd ? A.e41 : A.e31, eb = odd ? A.e42 : 0.0;
    double q = on * K.q0[i], s2 = on * A.p0[i], cq = 0.0, cp = 0.0;
    double Sm = 0.0, cS = 0.0, Un = 0.0;
    using Tb = aff::Table<double, M, FORCE>;
    const int n = K.n_steps;
    const double* row = tab;
    const double* end = tab + (size_t)(K.spc2 >> 1) * Tb::stride;
    auto term = [&](int k) -> double {
        if constexpr (Tb::compact)
            return ::fma(A.dS[k], row[0], A.dC[k] * row[1]);
        else
            return row[k];
    };
    for (int k = 0; k <= n; ++k) {
        // the sums of the step's start: stage gaps 1 and 2, and (as the output
        // of the previous step) the tip deflection
        double u1, t2 = aff::fma(g2p, s2, g2q * q);
        double gap = 0.0;
        if constexpr (rate) {
            u1 = group_sum64<L>(q);
        } else {
            u1 = group_sum64_split<L>(q, t2, odd);   // even lanes: the tip deflection
            gap = aff::add(K.Zc, u1);
        }
        if (k > 0) {
            if (defl != nullptr && owner) defl[(size_t)(k - 1) * P + p] = u1;
            if (U != nullptr) aff::misfit_add(Un, u1, Sm, cS);
        }
        if (k == n) break;
        if (U != nullptr) Un = U[k];
        const double tq = term(2 + i), tp = term(2 + M + i);
        const double t3 = aff::fma(g3p, s2, g3q * q), t4 = aff::fma(g4p, s2, g4q * q);
        double F[4];
        if constexpr (rate) {
            const double d1 = aff::add(K.Zc, u1);
            const double d2 = aff::add(K.Zc, group_sum64<L>(t2));
            const double b3 = aff::add(aff::add(K.Zc, term(0)), group_sum64<L>(t3));
            const double b4 = aff::add(aff::add(K.Zc, term(1)), group_sum64<L>(t4));
            const double r1 = group_sum64<L>(aff::fma(r1p, s2, r1q * q));
            double r2 = aff::add(term(2 + 2 * M), group_sum64<L>(aff::fma(r2p, s2, r2q * q)));
            double r3 = aff::add(term(3 + 2 * M), group_sum64<L>(aff::fma(r3p, s2, r3q * q)));
            double r4 = aff::add(term(4 + 2 * M), group_sum64<L>(aff::fma(r4p, s2, r4q * q)));
            F[0] = aff::law<FORCE, double>(c, d1, r1);
            r2 = aff::fma(A.h21, F[0], r2);
            F[1] = aff::law<FORCE, double>(c, d2, r2);
            r3 = aff::fma(A.h32, F[1], aff::fma(A.h31, F[0], r3));
            F[2] = aff::law<FORCE, double>(c, aff::fma(A.e31, F[0], b3), r3);
            r4 = aff::fma(A.h43, F[2], aff::fma(A.h42, F[1], aff::fma(A.h41, F[0], r4)));
            F[3] = aff::law<FORCE, double>(
                c, aff::fma(A.e42, F[1], aff::fma(A.e41, F[0], b4)), r4);
        } else {
            const double b = aff::add(aff::add(K.Zc, term(odd ? 1 : 0)),
                                      group_sum64_split<L>(t3, t4, odd));
            const double Fa = aff::law<FORCE, double>(c, gap, 0.0);
            const double Fb = __shfl_xor_sync(0xffffffffu, Fa, 1);
            F[0] = odd ? Fb : Fa;
            F[1] = odd ? Fa : Fb;
            const double d34 = aff::fma(eb, F[1], aff::fma(ea, F[0], b));
            const double Fc = aff::law<FORCE, double>(c, d34, 0.0);
            const double Fd = __shfl_xor_sync(0xffffffffu, Fc, 1);
            F[2] = odd ? Fd : Fc;
            F[3] = odd ? Fc : Fd;
        }
        double iq = aff::sub(real ? tq : 0.0, cq), ip = aff::sub(real ? tp : 0.0, cp);
        iq = aff::fma(A1, q, iq);
        ip = aff::fma(D1, s2, ip);
#pragma unroll
        for (int s = 0; s < 3; ++s) {
            iq = aff::fma(bq[s], F[s], iq);
            ip = aff::fma(bp[s], F[s], ip);
        }
        ip = aff::fma(bp[3], F[3], ip);
        iq = aff::fma(B, s2, iq);
        ip = aff::fma(Cq, q, ip);
        aff::comp_add(q, cq, iq);
        aff::comp_add(s2, cp, ip);
        row += Tb::stride;
        if (row == end) row = tab;
    }
    if (S != nullptr && owner) store_misfit64(Sm, S, p, flags);
}

cudaError_t launch_forward_f64(const KAffine<double>& K, const double* x, int P, double* defl,
                               const double* U, double* S, int* flags, cudaStream_t st) {
    return dispatch_mf(K.m, K.force, [&](auto Mc, auto Fc) -> cudaError_t {
        constexpr int M = decltype(Mc)::value, FORCE = decltype(Fc)::value;
        constexpr int G = 32 / Lanes64<M>::value;
        const size_t smem = aff_table_bytes<double, M, FORCE>(K.spc2);
        const int warps = (P + G - 1) / G;
        // several lanes per candidate while their warps have a sub-partition
        // each (one thread per candidate is cheaper in lane-operations); as
        // few warps per block as spread over the SMs
        const bool lanes = warps <= 152 * 4;
        auto kern1 = fwd64_kernel<M, FORCE>;
        auto kernL = fwd64_lanes_kernel<M, FORCE>;
        if (smem > 48 * 1024) {
            const cudaError_t e = lanes
                ? cudaFuncSetAttribute(kernL, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)
                : cudaFuncSetAttribute(kern1, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
            if (e != cudaSuccess) return e;
        }
        if (lanes) {
            const int wpb = (warps + 151) / 152;
            kernL<<<(warps + wpb - 1) / wpb, 128, smem, st>>>(K, x, P, wpb, defl, U, S, flags);
        } else {
            kern1<<<(P + 127) / 128, 128, smem, st>>>(K, x, P, defl, U, S, flags);
        }
        return cudaGetLastError();
    });
}

}  // namespace afm
