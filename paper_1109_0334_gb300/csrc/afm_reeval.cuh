// afm_reeval.cuh -- device pieces of the FP64 re-evaluation by multiple
// shooting in time (kern_reeval.cu: one winner; kern_reeval_batch.cu: one
// winner per pixel of a batch): the FP64 RK4 step with the stage force
// slopes recorded, its FP32 linearisation, and the launch dispatch.
#pragma once

#include <type_traits>

#include "afm_affine.cuh"
#include "afm_device.cuh"
#include "afm_launch.h"

namespace afm {
namespace reeval {

constexpr double kDefectTol = 1e-9;
constexpr int kSweeps = 2;
constexpr int kRec = 8;   // recorded floats per RK4 step: (dF/dd, dF/dd') x 4 stages

inline size_t a256(size_t n) { return (n + 255) & ~size_t(255); }

// State components of the kernels' template mode count for m modes.
inline int reeval_modes(int m) { return (m == 1 || m == 3) ? m : AFM_MAXM; }

__host__ __device__ inline int reeval_segments(int n_steps) { return (n_steps + AFM_SEG - 1) / AFM_SEG; }

template <typename F>
cudaError_t dispatch_m13(int m, int force, F&& f) {
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
    if (m >= 1 && m <= AFM_MAXM) return byF(std::integral_constant<int, AFM_MAXM>{});
    return cudaErrorInvalidValue;
}

// One FP64 RK4 step in the affine form (afm_affine.cuh), uncompensated: FP64
// needs no compensation over a segment.  R: the step's drive terms.  REC: the
// force slopes of each stage go to rec[k * 32], k = 2 * stage (+1 for the rate
// slope).
template <int M, int FORCE, bool REC>
__device__ __forceinline__ void step64(const KConst<double>& K, const aff::LawCoef<double>& c,
                                       const Coef<float>& cf, const double* R,
                                       aff::State<double, M, aff::NONE>& s, float* rec) {
    aff::Stages<double> g;
    aff::stages<double, M, FORCE, aff::NONE>(K, c, R, s, g);
    if constexpr (REC) {
#pragma unroll
        for (int st = 0; st < 4; ++st) {
            float Fd, Fr, Fc[4];
            force_partials<FORCE>(cf, (float)g.d[st], (float)g.r[st], Fd, Fr, Fc);
            rec[(2 * st) * 32] = Fd;
            rec[(2 * st + 1) * 32] = Fr;
        }
    }
    aff::advance<double, M, aff::NONE>(K, R, g.F, s);
}

// Drive terms of phase j.  COMPACT: tab holds the sine and cosine of each
// phase (2 spc doubles), else the rows of build_rows.
template <int M, int FORCE, bool COMPACT>
__device__ __forceinline__ void drive_terms(const KConst<double>& K, const double* tab, int j,
                                            double (&R)[aff::Rows<M, FORCE>::words]) {
    if constexpr (COMPACT)
        aff::phase_terms<M, FORCE>(K, tab[2 * j], tab[2 * j + 1], R);
    else
        aff::load_row<double, M, FORCE>(K, tab + (size_t)j * aff::Rows<M, FORCE>::words, R);
}

// The whole record by one thread: the fallback of both re-evaluations.
template <int M, int FORCE, bool COMPACT>
__device__ __forceinline__ double integrate64(const KConst<double>& K,
                                              const aff::LawCoef<double>& c, const double* tab,
                                              const float* __restrict__ U, int n) {
    aff::State<double, M, aff::ALL> s;
    aff::init<double, M, aff::ALL>(K, s);
    double S = 0.0, cS = 0.0;
    const int spc = K.spc2 >> 1;
    int j = 0;
    for (int t = 0; t < n; ++t) {
        double R[aff::Rows<M, FORCE>::words];
        drive_terms<M, FORCE, COMPACT>(K, tab, j, R);
        if (++j == spc) j = 0;
        aff::step<double, M, FORCE, aff::ALL>(K, c, R, s);
        if (K.np > 0) {
            for (int k = 0; k < K.np; ++k)
                aff::misfit_add((double)U[(size_t)t * K.np + k], aff::point_defl(K, k, s), S, cS);
        } else {
            aff::misfit_add((double)U[t], aff::tip(s), S, cS);
        }
    }
    return S;
}

// FP32 steps 0 .. n - 1 of the winner from rows in shared memory (every word
// once); the FP64 value of the state after every AFM_SEG-th step goes to
// Y[b][2m], b = 1 .. B - 1.  One warp's instruction stream bounds it (~130
// per step): a step's drive terms are loaded during the step before.
template <int M, int FORCE>
__device__ __forceinline__ void guess_starts(const KConst<float>& Kf, const KConst<double>& Kd,
                                             const Coef<float>& cf, const float* rows, int n,
                                             int B, double* Y) {
    constexpr int S2 = 2 * M, W = aff::Rows<M, FORCE>::words;
    const aff::LawCoef<float> c = aff::law_coef(cf);
    aff::State<float, M, aff::MODE0> s;
    aff::init<float, M, aff::MODE0>(Kf, s);
    const float* row = rows;
    const float* end = rows + (size_t)(Kf.spc2 >> 1) * W;
    float R[W];
    aff::load_row<float, M, FORCE>(Kf, row, R);
    int b = 1, next = AFM_SEG;
    for (int t = 0; t < n && b < B; ++t) {
        row += W;
        if (row == end) row = rows;
        float Rn[W];
        aff::load_row<float, M, FORCE>(Kf, row, Rn);
        aff::step<float, M, FORCE, aff::MODE0>(Kf, c, R, s);
#pragma unroll
        for (int k = 0; k < W; ++k) R[k] = Rn[k];
        if (t + 1 == next) {
            aff::export_state<float, M, aff::MODE0>(Kd, s, Y + (size_t)b * S2,
                                                    Y + (size_t)b * S2 + M);
            ++b;
            next += AFM_SEG;
        }
    }
}

// Linearised stage: da = dA/d(q, v) . (dq, dv) with the recorded slopes.
template <int M, int FORCE>
__device__ __forceinline__ void jvp_stage(const float* w2, const float* wq, const float* tip,
                                          const float* rec, int st, const float* dq,
                                          const float* dv, float* da) {
    float su = dq[0];
#pragma unroll
    for (int i = 1; i < M; ++i) su += dq[i];
    float dF = rec[(2 * st) * 32] * su;
    if (UsesRate<FORCE>::value) {
        float sv = dv[0];
#pragma unroll
        for (int i = 1; i < M; ++i) sv += dv[i];
        dF = fmaf(rec[(2 * st + 1) * 32], sv, dF);
    }
#pragma unroll
    for (int i = 0; i < M; ++i) {
        const float base = fmaf(-wq[i], dv[i], -w2[i] * dq[i]);
        da[i] = (M <= 4) ? base + dF : fmaf(tip[i], dF, base);
    }
}

// The RK4 step (stage form, in q and v) linearised about its recorded stages, applied to one
// tangent direction (dq, dv) in place.
template <int M, int FORCE>
__device__ __forceinline__ void jvp_step(const float* w2, const float* wq, const float* tip,
                                         const float* rec, float* dq, float* dv) {
    float a[M], qs[M], vs[M], Kq[M], Kv[M];
    jvp_stage<M, FORCE>(w2, wq, tip, rec, 0, dq, dv, a);
#pragma unroll
    for (int i = 0; i < M; ++i) {
        Kq[i] = dv[i];
        Kv[i] = a[i];
        qs[i] = fmaf(3.f, dv[i], dq[i]);
        vs[i] = fmaf(3.f, a[i], dv[i]);
    }
    jvp_stage<M, FORCE>(w2, wq, tip, rec, 1, qs, vs, a);
#pragma unroll
    for (int i = 0; i < M; ++i) {
        Kq[i] = fmaf(2.f, vs[i], Kq[i]);
        Kv[i] = fmaf(2.f, a[i], Kv[i]);
        qs[i] = fmaf(3.f, vs[i], dq[i]);
        vs[i] = fmaf(3.f, a[i], dv[i]);
    }
    jvp_stage<M, FORCE>(w2, wq, tip, rec, 2, qs, vs, a);
#pragma unroll
    for (int i = 0; i < M; ++i) {
        Kq[i] = fmaf(2.f, vs[i], Kq[i]);
        Kv[i] = fmaf(2.f, a[i], Kv[i]);
        qs[i] = fmaf(6.f, vs[i], dq[i]);
        vs[i] = fmaf(6.f, a[i], dv[i]);
    }
    jvp_stage<M, FORCE>(w2, wq, tip, rec, 3, qs, vs, a);
#pragma unroll
    for (int i = 0; i < M; ++i) {
        dq[i] = dq[i] + (Kq[i] + vs[i]);
        dv[i] = dv[i] + (Kv[i] + a[i]);
    }
}

__device__ __forceinline__ Coef<double> winner_coef(const ReevalWinner& w) {
    Coef<double> c;
    c.c0 = w.c[0];
    c.c1 = w.c[1];
    c.c2 = w.c[2];
    c.c3 = w.c[3];
    return c;
}

}  // namespace reeval
}  // namespace afm
