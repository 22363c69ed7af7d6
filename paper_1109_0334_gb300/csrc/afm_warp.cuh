// afm_warp.cuh -- the FP32 time loops for batches of at most one warp per SM
// sub-partition, one particle per lane.
//
// Such a launch takes as long as one warp's recurrence: ~150 FP32
// operations per step for three modes and the DMT law, issued in order along
// two force evaluations in series (~40 clocks each: min/max, special
// function, products).  What that warp must not do besides:
//   wait on global memory      the record is read 32 values at a time, a block
//                              ahead, one per lane, and handed out by a
//                              shuffle (a load per step pays the miss of every
//                              32nd step)
//   wait on shared memory      a step's drive values are loaded during the
//                              step before; gam g of the step's end is the
//                              next one's start
//   force after force          for rate-free laws stage 2's gap needs only
//                              q + (h/2) v and stage 4's only a_2, so F2 is
//                              formed before F1 and F4 before F3: their
//                              special functions overlap
//   branch every step          two steps per loop round (four for one or two
//                              modes; more ran slower)
// Measured per step (DMT, three modes): 98 ns.  One thread without these took
// 194 ns; spreading the modes over three lanes of a warp 151 ns (two rounds of
// shuffles in the chain of every step); the modes of a thread in paired FP32
// instructions 125 ns (one warp issues a paired instruction every two clocks).
//
// Every operation is rk4_step's, with the contractions that nvcc makes of it
// written out, so results are bit-identical to the throughput kernels'
// (afm_device.cuh, afm_f32x2.cuh).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

#include "afm_device.cuh"

namespace afm {
namespace warp {

// Modal constants with the signs accel uses, and the carried state.
template <int M>
struct Modes {
    float nwq[M], nw2[M], gam[M], tip[M], nw2lo, Zc;
};

template <int M>
__device__ __forceinline__ Modes<M> modes(const KConst<float>& K) {
    Modes<M> C;
#pragma unroll
    for (int i = 0; i < M; ++i) {
        C.nwq[i] = -K.wq[i];
        C.nw2[i] = -K.w2[i];
        C.gam[i] = K.gam[i];
        C.tip[i] = K.tip[i];
    }
    C.nw2lo = -K.w2lo[0];
    C.Zc = K.Zc;
    return C;
}

template <int M>
struct State {
    float q[M], v[M], gg[M];   // gg: gam g at the step's start
    float cq, cv, u;           // compensations of mode 0, tip deflection
};

template <int M>
__device__ __forceinline__ float sum(const float* a) {
    float u = a[0];
#pragma unroll
    for (int i = 1; i < M; ++i) u = __fadd_rn(u, a[i]);
    return u;
}

template <int M>
__device__ __forceinline__ void axpy(float s, const float* x, const float* y, float* r) {
#pragma unroll
    for (int i = 0; i < M; ++i) r[i] = __fmaf_rn(s, x[i], y[i]);
}

template <int M>
__device__ __forceinline__ void init(const KConst<float>& K, const Modes<M>& C, float g0,
                                     State<M>& s) {
#pragma unroll
    for (int i = 0; i < M; ++i) {
        s.q[i] = K.q0[i];
        s.v[i] = K.v0[i];
        s.gg[i] = __fmul_rn(C.gam[i], g0);
    }
    s.cq = s.cv = 0.f;
    s.u = sum<M>(s.q);
}

// tip_force in the form nvcc contracts it to.
template <int FORCE>
__device__ __forceinline__ float law(const Coef<float>& c, float d, float dd) {
    if constexpr (FORCE == F_LINEAR) {
        return __fmul_rn(-c.c0, __fsub_rn(d, c.c1));
    } else if constexpr (FORCE == F_DMT || FORCE == F_DMT_KV) {
        const float r = rcp_fast(fmaxf(d, c.c3));
        const float del = fmaxf(__fsub_rn(c.c3, d), 0.f);
        const float sq = sqrt_fast(del);
        float F = __fmaf_rn(c.c0, __fmul_rn(del, sq), -__fmul_rn(c.c1, __fmul_rn(r, r)));
        if constexpr (FORCE == F_DMT_KV) F = __fmaf_rn(-c.c2, __fmul_rn(sq, dd), F);
        return F;
    } else if constexpr (FORCE == F_HOOKE) {
        return __fmul_rn(c.c0, fmaxf(__fsub_rn(c.c1, d), 0.f));
    } else {
        return d < c.c1 ? __fmaf_rn(c.c0, __fsub_rn(c.c1, d), -__fmul_rn(c.c2, dd)) : 0.f;
    }
}

// accel of afm_device.cuh from the drive products and the tip force.
template <int M>
__device__ __forceinline__ void accel(const Modes<M>& C, const float* q, const float* v,
                                      const float* gg, float F, float* a) {
#pragma unroll
    for (int i = 0; i < M; ++i) {
        float ai = __fmaf_rn(C.nwq[i], v[i], gg[i]);
        if (i == 0) ai = __fmaf_rn(C.nw2lo, q[0], ai);
        ai = __fmaf_rn(C.nw2[i], q[i], ai);
        a[i] = M <= 4 ? __fadd_rn(ai, F) : __fmaf_rn(C.tip[i], F, ai);
    }
}

// Gaps and gap rates of a step's four stages.
struct Gaps {
    float d[4], r[4];
};

// One step (rk4_step); gh, g1: drive at t + h/2 and t + h; g: its stage gaps.
template <int M, int FORCE>
__device__ __forceinline__ void step(const Modes<M>& C, const Coef<float>& c, float gh, float g1,
                                     State<M>& s, Gaps& g) {
    float ggh[M], gg1[M], q2[M], q3[M], q4[M], v2[M], v3[M], v4[M], a1[M], a2[M], a3[M], a4[M];
#pragma unroll
    for (int i = 0; i < M; ++i) {
        ggh[i] = __fmul_rn(C.gam[i], gh);
        gg1[i] = __fmul_rn(C.gam[i], g1);
    }
    axpy<M>(3.f, s.v, s.q, q2);
    if constexpr (!UsesRate<FORCE>::value) {
        g.r[0] = g.r[1] = g.r[2] = g.r[3] = 0.f;
        g.d[1] = __fadd_rn(C.Zc, sum<M>(q2));
        g.d[0] = __fadd_rn(C.Zc, s.u);
        const float F2 = law<FORCE>(c, g.d[1], 0.f);
        const float F1 = law<FORCE>(c, g.d[0], 0.f);
        accel<M>(C, s.q, s.v, s.gg, F1, a1);
        axpy<M>(3.f, a1, s.v, v2);
        accel<M>(C, q2, v2, ggh, F2, a2);
        axpy<M>(3.f, v2, s.q, q3);
        axpy<M>(3.f, a2, s.v, v3);
        axpy<M>(6.f, v3, s.q, q4);
        g.d[3] = __fadd_rn(C.Zc, sum<M>(q4));
        g.d[2] = __fadd_rn(C.Zc, sum<M>(q3));
        const float F4 = law<FORCE>(c, g.d[3], 0.f);
        const float F3 = law<FORCE>(c, g.d[2], 0.f);
        accel<M>(C, q3, v3, ggh, F3, a3);
        axpy<M>(6.f, a3, s.v, v4);
        accel<M>(C, q4, v4, gg1, F4, a4);
    } else {
        g.d[0] = __fadd_rn(C.Zc, s.u);
        g.r[0] = sum<M>(s.v);
        const float F1 = law<FORCE>(c, g.d[0], g.r[0]);
        accel<M>(C, s.q, s.v, s.gg, F1, a1);
        axpy<M>(3.f, a1, s.v, v2);
        g.d[1] = __fadd_rn(C.Zc, sum<M>(q2));
        g.r[1] = sum<M>(v2);
        const float F2 = law<FORCE>(c, g.d[1], g.r[1]);
        accel<M>(C, q2, v2, ggh, F2, a2);
        axpy<M>(3.f, v2, s.q, q3);
        axpy<M>(3.f, a2, s.v, v3);
        g.d[2] = __fadd_rn(C.Zc, sum<M>(q3));
        g.r[2] = sum<M>(v3);
        const float F3 = law<FORCE>(c, g.d[2], g.r[2]);
        accel<M>(C, q3, v3, ggh, F3, a3);
        axpy<M>(6.f, v3, s.q, q4);
        axpy<M>(6.f, a3, s.v, v4);
        g.d[3] = __fadd_rn(C.Zc, sum<M>(q4));
        g.r[3] = sum<M>(v4);
        const float F4 = law<FORCE>(c, g.d[3], g.r[3]);
        accel<M>(C, q4, v4, gg1, F4, a4);
    }
#pragma unroll
    for (int i = 0; i < M; ++i) {
        float Kq = __fmaf_rn(2.f, v2[i], s.v[i]), Kv = __fmaf_rn(2.f, a2[i], a1[i]);
        Kq = __fadd_rn(__fmaf_rn(2.f, v3[i], Kq), v4[i]);
        Kv = __fadd_rn(__fmaf_rn(2.f, a3[i], Kv), a4[i]);
        state_add(i, s.q[i], s.cq, Kq);   // compensated for mode 0 only
        state_add(i, s.v[i], s.cv, Kv);
        s.gg[i] = gg1[i];
    }
    s.u = sum<M>(s.q);
}

template <int M, int FORCE>
__device__ __forceinline__ void step(const Modes<M>& C, const Coef<float>& c, float gh, float g1,
                                     State<M>& s) {
    Gaps g;
    step<M, FORCE>(C, c, gh, g1, s, g);
}

__device__ __forceinline__ void misfit_add(float U, float u, float& S, float& cS) {
    const float r = __fsub_rn(U, u);
    const float y = __fmaf_rn(r, r, -cS);
    const float t = __fadd_rn(S, y);
    cS = __fsub_rn(__fsub_rn(t, S), y);
    S = t;
}

// Particles of one warp per SM sub-partition (152 SMs x 4), and the particles
// per 128-thread block that spread a smaller batch over the SMs: 32 while
// every warp can have an SM of its own, up to 128 (the block's other warps
// help build the drive table and leave).
inline int max_particles() { return 152 * 4 * 32; }
inline int per_block(int P) {
    const int w = (P + 152 * 32 - 1) / (152 * 32);
    return 32 * (w < 1 ? 1 : w > 4 ? 4 : w);
}

// Template mode count for m modes: the modes past m have zero constants.
template <typename F>
cudaError_t dispatch(int m, int force, F&& f) {
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
    if (m == 2) return byF(std::integral_constant<int, 2>{});
    if (m == 3) return byF(std::integral_constant<int, 3>{});
    if (m <= 5) return byF(std::integral_constant<int, 5>{});
    return byF(std::integral_constant<int, AFM_MAXM>{});
}

}  // namespace warp

// integrate() (FP32) of one particle, for warps whose lanes all follow one
// record of n steps.  Every lane of the warp must call it; store: the lane's
// deflections are written.
template <int M, int FORCE>
__device__ __forceinline__ float integrate_warp(const KConst<float>& K, const Coef<float>& c,
                                                const float* tab, const float* __restrict__ U,
                                                float* __restrict__ defl, int P, int p, int n,
                                                bool store) {
    const warp::Modes<M> C = warp::modes<M>(K);
    warp::State<M> s;
    warp::init<M>(K, C, tab[0], s);
    float S = 0.f, cS = 0.f;
    const int lane = threadIdx.x & 31, spc2 = K.spc2;
    int j = 0;
    float gh = tab[1], g1 = tab[2];
    float Ub = (U != nullptr && lane < n) ? U[lane] : 0.f;
    auto one = [&](int k0, int k) {
        j += 2;
        if (j >= spc2) j = 0;
        const float ghn = tab[j + 1], g1n = tab[j + 2];
        const float Un = __shfl_sync(0xffffffffu, Ub, k);
        warp::step<M, FORCE>(C, c, gh, g1, s);
        if (defl != nullptr && store) defl[(size_t)(k0 + k) * P + p] = s.u;
        warp::misfit_add(Un, s.u, S, cS);
        gh = ghn;
        g1 = g1n;
    };
    constexpr int UNROLL = M <= 2 ? 4 : 2;
    for (int k0 = 0; k0 < n; k0 += 32) {
        const int kn = k0 + 32 + lane;
        const float Unb = (U != nullptr && kn < n) ? U[kn] : 0.f;
        if (k0 + 32 <= n) {
#pragma unroll UNROLL
            for (int k = 0; k < 32; ++k) one(k0, k);
        } else {
            for (int k = 0; k < n - k0; ++k) one(k0, k);
        }
        Ub = Unb;
    }
    return S;
}

// The same over the deflection points (integrate_points, misfit only), any
// lanes: the record values of a step are loaded during the step before.  The
// point count is a constant of the loop: 512 particles x 4096 steps x 3
// points, nine launches and the re-evaluation, 5.86 ms, 8.63 with the points
// under a uniform guard.
template <int M, int FORCE, int NP>
__device__ __forceinline__ float integrate_points_of(const KConst<float>& K,
                                                     const Coef<float>& c, const float* tab,
                                                     const float* __restrict__ U, int n) {
    const warp::Modes<M> C = warp::modes<M>(K);
    warp::State<M> s;
    warp::init<M>(K, C, tab[0], s);
    float S = 0.f, cS = 0.f;
    const int spc2 = K.spc2;
    int j = 0;
    float gh = tab[1], g1 = tab[2];
    float Ucur[NP];
#pragma unroll
    for (int k = 0; k < NP; ++k) Ucur[k] = n > 0 ? U[k] : 0.f;
#pragma unroll 2
    for (int t = 0; t < n; ++t) {
        j += 2;
        if (j >= spc2) j = 0;
        const float ghn = tab[j + 1], g1n = tab[j + 2];
        const float* Un = U + (size_t)min(t + 1, n - 1) * NP;
        float Unext[NP];
#pragma unroll
        for (int k = 0; k < NP; ++k) Unext[k] = Un[k];
        warp::step<M, FORCE>(C, c, gh, g1, s);
#pragma unroll
        for (int k = 0; k < NP; ++k) {
            float uk = __fmul_rn(K.phi[k][0], s.q[0]);
#pragma unroll
            for (int i = 1; i < M; ++i) uk = __fmaf_rn(K.phi[k][i], s.q[i], uk);
            warp::misfit_add(Ucur[k], uk, S, cS);
        }
#pragma unroll
        for (int k = 0; k < NP; ++k) Ucur[k] = Unext[k];
        gh = ghn;
        g1 = g1n;
    }
    return S;
}

template <int M, int FORCE>
__device__ __forceinline__ float integrate_points_warp(const KConst<float>& K,
                                                       const Coef<float>& c, const float* tab,
                                                       const float* __restrict__ U, int n) {
    static_assert(AFM_MAX_POINTS == 4, "a loop per point count");
    switch (K.np) {
        case 1: return integrate_points_of<M, FORCE, 1>(K, c, tab, U, n);
        case 2: return integrate_points_of<M, FORCE, 2>(K, c, tab, U, n);
        case 3: return integrate_points_of<M, FORCE, 3>(K, c, tab, U, n);
        default: return integrate_points_of<M, FORCE, 4>(K, c, tab, U, n);
    }
}

}  // namespace afm
