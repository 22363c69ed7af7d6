// afm_affine.cuh -- one classic RK4 step of the modal cantilever (Eq. 2,
// Sec. 3.2) in its affine form (struct Affine of afm_internal.h): the stage
// states themselves are never formed, only the four stage gaps and the
// increments, 97 operations per particle and step for three modes and the
// DMT law where the stages evaluated mode by mode take 147.  For rate-free
// laws F1 and F2 depend on the step's start state only and F3 and F4 on them
// through one fma each, so a step is two force evaluations deep.
//
// Used by the FP64 solves (kern_forward64.cu, the passes of afm_reeval.cuh),
// the tangents (afm_tangent.cuh), the adjoint of few particles
// (kern_adjoint.cu) and the FP32 guesses of the re-evaluation.
// The FP32 forward solves keep the stage form of afm_device.cuh: in FP32 the
// two forms round differently, and a swarm's misfits would move by up to
// 5e-5 of their value near the noise floor (the stage form's own distance
// from FP64 there; the affine form is two to three times closer).
//
// Rounding: the small terms of a sum come first and the state's own term
// last (a small force added to a large partial sum is rounded with a bias
// that the resonance accumulates).  Every operation is written out (no
// contraction is left to the compiler).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

#include "afm_device.cuh"

namespace afm {
namespace aff {

// ---- operations, float and double ----------------------------------------------
__device__ __forceinline__ float add(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float sub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float mul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float fma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ float neg(float a) { return -a; }
__device__ __forceinline__ float vmax(float a, float b) { return fmaxf(a, b); }
__device__ __forceinline__ float vrcp(float a) { return rcp_fast(a); }
__device__ __forceinline__ float vsqrt(float a) { return sqrt_fast(a); }

__device__ __forceinline__ double add(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ double sub(double a, double b) { return __dsub_rn(a, b); }
__device__ __forceinline__ double mul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ double fma(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ double neg(double a) { return -a; }
__device__ __forceinline__ double vmax(double a, double b) { return fmax(a, b); }

// ---- tip-sample laws ---------------------------------------------------------
template <typename V>
struct LawCoef {
    V c0, c1, c2, c3;
    V vc;   // the DMT contact branch's van der Waals term c1 / a0^2
};

template <typename T>
__device__ __forceinline__ LawCoef<T> law_coef(const Coef<T>& a) {
    LawCoef<T> c;
    c.c0 = a.c0;
    c.c1 = a.c1;
    c.c2 = a.c2;
    c.c3 = a.c3;
    const T r = rcp_fast(a.c3);
    c.vc = mul(a.c1, mul(r, r));
    return c;
}

template <int FORCE, typename V>
__device__ __forceinline__ V law(const LawCoef<V>& c, V d, V dd) {
    if constexpr (FORCE == F_LINEAR) {
        return mul(neg(c.c0), sub(d, c.c1));
    } else if constexpr ((FORCE == F_DMT || FORCE == F_DMT_KV) && sizeof(V) == 8) {
        // FP64: a reciprocal out of contact or a square root in it, not both
        // (each is a sequence of FP64 operations at 64 clocks a warp).  The
        // van der Waals term of the contact branch is its value at d = a0.
        if (d < c.c3) {
            const V del = sub(c.c3, d), sq = sqrt_fast(del);
            V F = fma(c.c0, mul(del, sq), neg(c.vc));
            if constexpr (FORCE == F_DMT_KV) F = fma(neg(c.c2), mul(sq, dd), F);
            return F;
        }
        const V r = rcp_fast(d);
        return neg(mul(c.c1, mul(r, r)));
    } else if constexpr (FORCE == F_DMT || FORCE == F_DMT_KV) {
        // branch-free: the van der Waals term saturates at d = a0, where it is
        // the contact branch's constant
        const V r = vrcp(vmax(d, c.c3));
        const V del = vmax(sub(c.c3, d), (V)0);
        const V sq = vsqrt(del);
        V F = fma(c.c0, mul(del, sq), neg(mul(c.c1, mul(r, r))));
        if constexpr (FORCE == F_DMT_KV) F = fma(neg(c.c2), mul(sq, dd), F);
        return F;
    } else if constexpr (FORCE == F_HOOKE) {
        return mul(c.c0, vmax(sub(c.c1, d), (V)0));
    } else {
        return d < c.c1 ? fma(c.c0, sub(c.c1, d), neg(mul(c.c2, dd))) : (V)0;
    }
}

// ---- drive-term rows ---------------------------------------------------------
template <int M, int FORCE>
struct Rows {
    static constexpr bool rate = UsesRate<FORCE>::value;
    static constexpr int terms = 2 + 2 * M + (rate ? 3 : 0);
    static constexpr int words = aff_row(M, rate);
};

// Table words per phase.  FP64 with 8 modes keeps the sine and cosine of the
// phase and forms the terms in each step (20 or 24 doubles for each of up to
// 2048 phases would not fit shared memory; 36 of ~400 FP64 operations a
// step).
template <typename T, int M, int FORCE>
struct Table {
    static constexpr bool compact = sizeof(T) == 8 && M > 3;
    static constexpr int stride = compact ? 2 : Rows<M, FORCE>::words;
};

// The drive terms of every phase of the period, evaluated in FP64 by the
// block's threads.
template <typename T, int M, int FORCE>
__device__ __forceinline__ void build_rows(const KAffine<T>& K, T* tab) {
    using R = Rows<M, FORCE>;
    using Tb = Table<T, M, FORCE>;
    const int spc = K.spc2 >> 1;
    const double step = 2.0 / (double)spc;
    for (int j = threadIdx.x; j < spc; j += blockDim.x) {
        double s, c;
        sincospi(step * (double)j, &s, &c);
        T* row = tab + (size_t)j * Tb::stride;
        if constexpr (Tb::compact) {
            row[0] = s;
            row[1] = c;
        } else {
#pragma unroll
            for (int k = 0; k < R::words; ++k)
                row[k] = k < R::terms ? (T)::fma(K.af.dS[k], s, K.af.dC[k] * c) : (T)0;
        }
    }
}

// The terms of a phase from its sine and cosine.
template <int M, int FORCE>
__device__ __forceinline__ void phase_terms(const KAffine<double>& K, double s, double c,
                                            double (&r)[Rows<M, FORCE>::words]) {
#pragma unroll
    for (int k = 0; k < Rows<M, FORCE>::words; ++k)
        r[k] = k < Rows<M, FORCE>::terms ? ::fma(K.af.dS[k], s, K.af.dC[k] * c) : 0.0;
}

// One row into registers, 16 bytes per load.
template <typename T, int M, int FORCE>
__device__ __forceinline__ void load_row(const KAffine<T>& K, const T* __restrict__ row,
                                         T (&r)[Rows<M, FORCE>::words]) {
    constexpr int WORDS = Rows<M, FORCE>::words;
    static_assert(WORDS % 4 == 0, "16-byte rows");
    if constexpr (Table<T, M, FORCE>::compact) {
        phase_terms<M, FORCE>(K, row[0], row[1], r);
    } else if constexpr (sizeof(T) == 4) {
        const float4* p = reinterpret_cast<const float4*>(row);
#pragma unroll
        for (int k = 0; k < WORDS / 4; ++k) {
            const float4 t = p[k];
            r[4 * k] = t.x;
            r[4 * k + 1] = t.y;
            r[4 * k + 2] = t.z;
            r[4 * k + 3] = t.w;
        }
    } else {
        const double2* p = reinterpret_cast<const double2*>(row);
#pragma unroll
        for (int k = 0; k < WORDS / 2; ++k) {
            const double2 t = p[k];
            r[2 * k] = t.x;
            r[2 * k + 1] = t.y;
        }
    }
}

// ---- state and step ----------------------------------------------------------
// COMP: which modes take compensated updates.  s1 is the sum of the
// deflections of modes >= 1 (the tip deflection is q[0] + s1).
enum Comp { NONE = 0, MODE0 = 1, ALL = 2 };
template <typename V, int M, int COMP>
struct State {
    V q[M], p[M], s1;
    V cq[COMP == ALL ? M : 1], cp[COMP == ALL ? M : 1];
};

template <typename V, int M>
__device__ __forceinline__ V sum_tail(const V* a) {   // a[1] + a[2] + ...
    V s = (V)0;
    if constexpr (M > 1) {
        s = a[1];
#pragma unroll
        for (int i = 2; i < M; ++i) s = add(s, a[i]);
    }
    return s;
}

template <typename V, int M, int COMP, typename T>
__device__ __forceinline__ void init(const KAffine<T>& K, State<V, M, COMP>& s) {
#pragma unroll
    for (int i = 0; i < M; ++i) {
        s.q[i] = K.q0[i];
        s.p[i] = K.af.p0[i];
    }
#pragma unroll
    for (int i = 0; i < (COMP == ALL ? M : 1); ++i) s.cq[i] = s.cp[i] = (V)0;
    s.s1 = sum_tail<V, M>(s.q);
}

template <typename V, int M, int COMP>
__device__ __forceinline__ V tip(const State<V, M, COMP>& s) {
    if constexpr (M > 1)
        return add(s.q[0], s.s1);
    else
        return s.q[0];
}

// x += y - c (the compensation is already inside y), new compensation c.
template <typename V>
__device__ __forceinline__ void comp_add(V& x, V& c, V y) {
    const V t = add(x, y);
    c = sub(sub(t, x), y);
    x = t;
}

template <bool COMPENSATED, typename V>
__device__ __forceinline__ void update(V& x, V& c, V y) {
    if constexpr (COMPENSATED)
        comp_add(x, c, y);
    else
        x = add(x, y);
}

// Gaps (and gap rates) and forces of the four stages of one step.
template <typename V>
struct Stages {
    V d[4], F[4], r[4];
};

template <typename V, int M, int FORCE, int COMP, typename T>
__device__ __forceinline__ void stages(const KAffine<T>& K, const LawCoef<V>& c, const V* R,
                                       const State<V, M, COMP>& s, Stages<V>& g) {
    const Affine<T>& A = K.af;
    constexpr bool rate = UsesRate<FORCE>::value;
    // the gap is the small difference of Zc and q_0: in FP32 with every mode
    // compensated (the adjoint) it takes q_0's lost bits, on which contact
    // events and their slopes hang
    V zq = add(K.Zc, s.q[0]);
    if constexpr (COMP == ALL && sizeof(V) == 4) zq = sub(zq, s.cq[0]);
    g.d[0] = M > 1 ? add(zq, s.s1) : zq;
    V sp = (V)0, a;
    if constexpr (M > 1) {
        sp = sum_tail<V, M>(s.p);
        a = fma(A.d2q, s.q[0], add(sp, s.s1));
    } else {
        a = mul(A.d2q, s.q[0]);
    }
    a = fma(A.d2w, s.p[0], a);
    g.d[1] = add(zq, a);
    V a3 = R[0], a4 = R[1];
#pragma unroll
    for (int i = 1; i < M; ++i) {
        a3 = fma(A.d3q[i], s.q[i], a3);
        a3 = fma(A.d3p[i], s.p[i], a3);
        a4 = fma(A.d4q[i], s.q[i], a4);
        a4 = fma(A.d4p[i], s.p[i], a4);
    }
    a3 = fma(A.d3q[0], s.q[0], a3);
    a3 = fma(A.d3p[0], s.p[0], a3);
    a4 = fma(A.d4q[0], s.q[0], a4);
    a4 = fma(A.d4p[0], s.p[0], a4);
    const V b3 = add(zq, a3), b4 = add(zq, a4);
    V r2 = (V)0, r3 = (V)0, r4 = (V)0;
    g.r[0] = g.r[1] = g.r[2] = g.r[3] = (V)0;
    if constexpr (rate) {
        g.r[0] = fma(A.v1w, s.p[0], mul(A.v1q, s.q[0]));
        if constexpr (M > 1) g.r[0] = fma(A.third, sp, g.r[0]);
        r2 = R[2 + 2 * M];
        r3 = R[3 + 2 * M];
        r4 = R[4 + 2 * M];
#pragma unroll
        for (int i = M - 1; i >= 0; --i) {
            r2 = fma(A.r2q[i], s.q[i], r2);
            r2 = fma(A.r2p[i], s.p[i], r2);
            r3 = fma(A.r3q[i], s.q[i], r3);
            r3 = fma(A.r3p[i], s.p[i], r3);
            r4 = fma(A.r4q[i], s.q[i], r4);
            r4 = fma(A.r4p[i], s.p[i], r4);
        }
    }
    g.F[0] = law<FORCE, V>(c, g.d[0], g.r[0]);
    if constexpr (rate) g.r[1] = fma(A.h21, g.F[0], r2);
    g.F[1] = law<FORCE, V>(c, g.d[1], g.r[1]);
    g.d[2] = fma(A.e31, g.F[0], b3);
    if constexpr (rate) g.r[2] = fma(A.h32, g.F[1], fma(A.h31, g.F[0], r3));
    g.F[2] = law<FORCE, V>(c, g.d[2], g.r[2]);
    g.d[3] = fma(A.e42, g.F[1], fma(A.e41, g.F[0], b4));
    if constexpr (rate)
        g.r[3] = fma(A.h43, g.F[2],
                     fma(A.h42, g.F[1], fma(A.h41, g.F[0], r4)));
    g.F[3] = law<FORCE, V>(c, g.d[3], g.r[3]);
}

// The step's increments from its four stage forces.
template <typename V, int M, int COMP, typename T>
__device__ __forceinline__ void advance(const KAffine<T>& K, const V* R, const V* F,
                                        State<V, M, COMP>& s) {
    const Affine<T>& A = K.af;
    {
        V iq = COMP ? sub(R[2], s.cq[0]) : R[2];
        iq = fma(A.bq[0][0], F[0], iq);
        iq = fma(A.bq[1][0], F[1], iq);
        iq = fma(A.bq[2][0], F[2], iq);
        iq = add(s.p[0], iq);
        const V qw = add(s.q[0], s.p[0]);
        V iw = COMP ? sub(R[2 + M], s.cp[0]) : R[2 + M];
        iw = fma(A.ec, s.p[0], iw);
        iw = fma(A.c0lo, qw, iw);
        iw = fma(A.bp[0][0], F[0], iw);
        iw = fma(A.bp[1][0], F[1], iw);
        iw = fma(A.bp[2][0], F[2], iw);
        iw = fma(A.bp[3][0], F[3], iw);
        iw = fma(A.c0, qw, iw);
        update<COMP != NONE>(s.q[0], s.cq[0], iq);
        update<COMP != NONE>(s.p[0], s.cp[0], iw);
    }
#pragma unroll
    for (int i = 1; i < M; ++i) {
        V iq = COMP == ALL ? sub(R[2 + i], s.cq[COMP == ALL ? i : 0]) : R[2 + i];
        V ip = COMP == ALL ? sub(R[2 + M + i], s.cp[COMP == ALL ? i : 0]) : R[2 + M + i];
        iq = fma(A.B[i], s.p[i], iq);
        iq = fma(A.A1[i], s.q[i], iq);
        ip = fma(A.D1[i], s.p[i], ip);
        ip = fma(A.C[i], s.q[i], ip);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            iq = fma(A.bq[k][i], F[k], iq);
            ip = fma(A.bp[k][i], F[k], ip);
        }
        ip = fma(A.bp[3][i], F[3], ip);
        update<COMP == ALL>(s.q[i], s.cq[COMP == ALL ? i : 0], iq);
        update<COMP == ALL>(s.p[i], s.cp[COMP == ALL ? i : 0], ip);
    }
    s.s1 = sum_tail<V, M>(s.q);
}

template <typename V, int M, int FORCE, int COMP, typename T>
__device__ __forceinline__ void step(const KAffine<T>& K, const LawCoef<V>& c, const V* R,
                                     State<V, M, COMP>& s) {
    Stages<V> g;
    stages<V, M, FORCE, COMP>(K, c, R, s, g);
    advance<V, M, COMP>(K, R, g.F, s);
}

// Compensated S += (U - u)^2.
template <typename V>
__device__ __forceinline__ void misfit_add(V U, V u, V& S, V& cS) {
    const V r = sub(U, u);
    const V y = fma(r, r, neg(cS));
    const V t = add(S, y);
    cS = sub(sub(t, S), y);
    S = t;
}

// Deflection at point k of the cantilever (K.phi), in the order of tip(), so
// that a point at the tip gives the tip's bits.
template <typename V, int M, int COMP, typename T>
__device__ __forceinline__ V point_defl(const KAffine<T>& K, int k, const State<V, M, COMP>& s) {
    if constexpr (M > 1) {
        V t = mul(K.phi[k][1], s.q[1]);
#pragma unroll
        for (int i = 2; i < M; ++i) t = fma(K.phi[k][i], s.q[i], t);
        return fma(K.phi[k][0], s.q[0], t);
    } else {
        return mul(K.phi[k][0], s.q[0]);
    }
}

// The state as (deflections, rates per tau) in FP64, compensations included.
template <typename T, int M, int COMP>
__device__ __forceinline__ void export_state(const KAffine<double>& K, const State<T, M, COMP>& s,
                                             double* q, double* v) {
#pragma unroll
    for (int i = 0; i < M; ++i) {
        const bool cmp = COMP == ALL || (COMP == MODE0 && i == 0);
        q[i] = (double)s.q[i] - (cmp ? (double)s.cq[COMP == ALL ? i : 0] : 0.0);
        const double p = (double)s.p[i] - (cmp ? (double)s.cp[COMP == ALL ? i : 0] : 0.0);
        v[i] = i == 0 ? ::fma(K.af.v1w, p, K.af.v1q * q[0]) : p * K.af.third;
    }
}

// ... and from them (uncompensated).
template <int M>
__device__ __forceinline__ void import_state(const KAffine<double>& K, const double* q,
                                             const double* v, State<double, M, NONE>& s) {
#pragma unroll
    for (int i = 0; i < M; ++i) {
        s.q[i] = q[i];
        s.p[i] = i == 0 ? ::fma(-K.af.v1q, q[0], v[0]) / K.af.v1w : 3.0 * v[i];
    }
    s.cq[0] = s.cp[0] = 0.0;
    s.s1 = sum_tail<double, M>(s.q);
}

}  // namespace aff

// Dynamic shared memory of the drive-term rows.
template <typename T, int M, int FORCE>
size_t aff_table_bytes(int spc2) {
    return sizeof(T) * (size_t)(spc2 >> 1) * aff::Table<T, M, FORCE>::stride;
}

}  // namespace afm
