// afm_tangent.cuh -- tangent-linear (forward-mode) form of the affine RK4 step
// (afm_affine.cuh) for the sensitivity kernels of kern_lm.cu and
// kern_lm_lanes.cu.
//
// The primal solve is the forward kernels' (afm_warp.cuh), which leaves the
// gaps of a step's four stages; about them the step is affine in the state
// and the four stage forces, so a tangent takes that map without the drive
// terms, with dF_s = Fd_s dd_s (+ Fr_s dr_s) + G_s: ~65 FP32 operations per
// direction and step for three modes, 112 when each stage's modal
// accelerations are linearised.
//
// Directions.  A force law has few coefficients (DMT: c0, c1, c3), its
// parameters enter only through them, and J = dc/dx is constant along a
// solve.  With at least as many free parameters as coefficients the
// tangents run along the coefficients themselves ("coefficient directions":
// G_s is one partial, no products) and the normal equations are mapped to
// the parameters once at the end, in FP64: H = J^T Hc J, b = J^T bc.  DMT
// with 4 unknowns carries 3 directions instead of 4, Kelvin-Voigt with 5
// carries 4.
#pragma once

#include "afm_affine.cuh"

namespace afm {
namespace aff {

// The law's coefficients (indices into c0..c3).
template <int FORCE>
struct CoefDirs {
    static constexpr int n = FORCE == F_DMT_KV ? 4
                             : (FORCE == F_DMT || FORCE == F_SPRING_DAMPER) ? 3 : 2;
    __host__ __device__ static constexpr int index(int k) {
        return FORCE == F_DMT && k == 2 ? 3 : k;
    }
};

// Partial derivatives of the tip force at one stage by the gap, its rate and
// the law's coefficients.
template <int FORCE>
struct Partials {
    float Fd, Fr, Fc[CoefDirs<FORCE>::n];
};

template <int FORCE>
__device__ __forceinline__ void partials(const Coef<float>& c, float d, float dd,
                                         Partials<FORCE>& P) {
    P.Fr = 0.f;
    if constexpr (FORCE == F_LINEAR) {
        P.Fd = -c.c0;
        P.Fc[0] = neg(sub(d, c.c1));
        P.Fc[1] = c.c0;
    } else if constexpr (FORCE == F_DMT || FORCE == F_DMT_KV) {
        const bool contact = d < c.c3;
        const float r = vrcp(fmaxf(d, c.c3));
        const float del = fmaxf(sub(c.c3, d), 0.f);
        const float sq = vsqrt(del);
        const float r2 = mul(r, r);
        const float hz = mul(mul(1.5f, c.c0), sq);          // zero out of contact
        const float vw = mul(mul(2.f, c.c1), mul(r2, r));
        P.Fd = contact ? -hz : vw;
        P.Fc[0] = mul(del, sq);
        P.Fc[1] = -r2;
        float Fa = contact ? add(hz, vw) : 0.f;
        if constexpr (FORCE == F_DMT_KV) {
            const float half = contact ? mul(mul(0.5f, mul(c.c2, dd)), vrcp(sq)) : 0.f;
            P.Fd = add(P.Fd, half);
            P.Fr = -mul(c.c2, sq);
            P.Fc[2] = -mul(sq, dd);
            Fa = sub(Fa, half);
        }
        P.Fc[CoefDirs<FORCE>::n - 1] = Fa;
    } else if constexpr (FORCE == F_HOOKE) {
        const bool contact = d < c.c1;
        P.Fd = contact ? -c.c0 : 0.f;
        P.Fc[0] = contact ? sub(c.c1, d) : 0.f;
        P.Fc[1] = contact ? c.c0 : 0.f;
    } else {
        const bool contact = d < c.c1;
        P.Fd = contact ? -c.c0 : 0.f;
        P.Fr = contact ? -c.c2 : 0.f;
        P.Fc[0] = contact ? sub(c.c1, d) : 0.f;
        P.Fc[1] = contact ? c.c0 : 0.f;
        P.Fc[2] = contact ? -dd : 0.f;
    }
}

// One tangent direction: derivatives of the state (plain sums) and s1, the
// sum over the modes >= 1 of the deflections' derivatives.
template <int M>
struct Tangent {
    float q[M], p[M], s1;
};

template <int M>
__device__ __forceinline__ void zero(Tangent<M>& t) {
#pragma unroll
    for (int i = 0; i < M; ++i) t.q[i] = t.p[i] = 0.f;
    t.s1 = 0.f;
}

template <int M>
__device__ __forceinline__ float tip(const Tangent<M>& t) {
    return M > 1 ? add(t.q[0], t.s1) : t.q[0];
}

// One step of a direction with the primal step's partials P[4] and the
// direction's own force terms G[4].
template <int M, int FORCE>
__device__ __forceinline__ void tangent_step(const KAffine<float>& K, const Partials<FORCE>* P,
                                             const float* G, Tangent<M>& t) {
    const Affine<float>& A = K.af;
    constexpr bool rate = UsesRate<FORCE>::value;
    const float e1 = tip(t);
    float sp = 0.f, a2 = mul(A.d2q, t.q[0]);
    if constexpr (M > 1) {
        sp = sum_tail<float, M>(t.p);
        a2 = add(sp, a2);
    }
    const float e2 = add(e1, fma(A.d2w, t.p[0], a2));
    float a3 = mul(A.d3p[0], t.p[0]), a4 = mul(A.d4p[0], t.p[0]);
    a3 = fma(A.d3q[0], t.q[0], a3);
    a4 = fma(A.d4q[0], t.q[0], a4);
#pragma unroll
    for (int i = 1; i < M; ++i) {
        a3 = fma(A.d3p[i], t.p[i], a3);
        a3 = fma(A.d3q[i], t.q[i], a3);
        a4 = fma(A.d4p[i], t.p[i], a4);
        a4 = fma(A.d4q[i], t.q[i], a4);
    }
    const float b3 = add(t.q[0], a3), b4 = add(t.q[0], a4);
    float r1 = 0.f, r2 = 0.f, r3 = 0.f, r4 = 0.f;
    if constexpr (rate) {
        r1 = fma(A.v1w, t.p[0], mul(A.v1q, t.q[0]));
        if constexpr (M > 1) r1 = fma(A.third, sp, r1);
#pragma unroll
        for (int i = M - 1; i >= 0; --i) {
            r2 = fma(A.r2q[i], t.q[i], r2);
            r2 = fma(A.r2p[i], t.p[i], r2);
            r3 = fma(A.r3q[i], t.q[i], r3);
            r3 = fma(A.r3p[i], t.p[i], r3);
            r4 = fma(A.r4q[i], t.q[i], r4);
            r4 = fma(A.r4p[i], t.p[i], r4);
        }
    }
    float F[4];
    auto dforce = [&](int s, float e, float r) {
        const float f = fma(P[s].Fd, e, G[s]);
        return rate ? fma(P[s].Fr, r, f) : f;
    };
    F[0] = dforce(0, e1, r1);
    if constexpr (rate) r2 = fma(A.h21, F[0], r2);
    F[1] = dforce(1, e2, r2);
    if constexpr (rate) r3 = fma(A.h32, F[1], fma(A.h31, F[0], r3));
    F[2] = dforce(2, fma(A.e31, F[0], b3), r3);
    if constexpr (rate) r4 = fma(A.h43, F[2], fma(A.h42, F[1], fma(A.h41, F[0], r4)));
    F[3] = dforce(3, fma(A.e42, F[1], fma(A.e41, F[0], b4)), r4);
    {
        float iq = mul(A.bq[0][0], F[0]);
        iq = fma(A.bq[1][0], F[1], iq);
        iq = fma(A.bq[2][0], F[2], iq);
        iq = add(t.p[0], iq);
        const float qw = add(t.q[0], t.p[0]);
        float iw = mul(A.ec, t.p[0]);
        iw = fma(A.c0lo, qw, iw);
#pragma unroll
        for (int k = 0; k < 4; ++k) iw = fma(A.bp[k][0], F[k], iw);
        iw = fma(A.c0, qw, iw);
        t.q[0] = add(t.q[0], iq);
        t.p[0] = add(t.p[0], iw);
    }
#pragma unroll
    for (int i = 1; i < M; ++i) {
        float iq = mul(A.B[i], t.p[i]), ip = mul(A.D1[i], t.p[i]);
        iq = fma(A.A1[i], t.q[i], iq);
        ip = fma(A.C[i], t.q[i], ip);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            iq = fma(A.bq[k][i], F[k], iq);
            ip = fma(A.bp[k][i], F[k], ip);
        }
        ip = fma(A.bp[3][i], F[3], ip);
        t.q[i] = add(t.q[i], iq);
        t.p[i] = add(t.p[i], ip);
    }
    t.s1 = sum_tail<float, M>(t.q);
}

// Row e of the parameters' normal equations from the coefficients': Hc is the
// lower triangle, entry (k, l <= k) at k (k + 1) / 2 + l.  Every kernel maps
// with this function, so their results agree bit for bit.
template <int NC>
__device__ __forceinline__ double hc_at(const double* Hc, int k, int l) {
    return k >= l ? Hc[k * (k + 1) / 2 + l] : Hc[l * (l + 1) / 2 + k];
}
template <int FORCE>
__device__ __forceinline__ void map_row(const double (&J)[4][AFM_MAXD], const double* Hc,
                                        const double* bc, int D, int e, double* H, double* b) {
    constexpr int NC = CoefDirs<FORCE>::n;
    double T[NC], be = 0.0;
#pragma unroll
    for (int l = 0; l < NC; ++l) T[l] = 0.0;
#pragma unroll
    for (int k = 0; k < NC; ++k) {
        const double Jke = J[CoefDirs<FORCE>::index(k)][e];
        be = ::fma(Jke, bc[k], be);
#pragma unroll
        for (int l = 0; l < NC; ++l) T[l] = ::fma(Jke, hc_at<NC>(Hc, k, l), T[l]);
    }
    b[e] = be;
    for (int g = 0; g <= e; ++g) {
        double h = 0.0;
#pragma unroll
        for (int l = 0; l < NC; ++l) h = ::fma(T[l], J[CoefDirs<FORCE>::index(l)][g], h);
        H[e * D + g] = h;
        H[g * D + e] = h;
    }
}

}  // namespace aff
}  // namespace afm
