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
__device__ __forceinline__ void step64(const KAffine<double>& K, const aff::LawCoef<double>& c,
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
__device__ __forceinline__ void drive_terms(const KAffine<double>& K, const double* tab, int j,
                                            double (&R)[aff::Rows<M, FORCE>::words]) {
    if constexpr (COMPACT)
        aff::phase_terms<M, FORCE>(K, tab[2 * j], tab[2 * j + 1], R);
    else
        aff::load_row<double, M, FORCE>(K, tab + (size_t)j * aff::Rows<M, FORCE>::words, R);
}

// The whole record by one thread: the fallback of both re-evaluations.
template <int M, int FORCE, bool COMPACT>
__device__ __forceinline__ double integrate64(const KAffine<double>& K,
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

// FP32 steps of the winner from rows in shared memory (every word once); the
// state after every AFM_SEG-th step goes to Y[b][2m], b = 1 .. B - 1, as
// (value, compensation) for finish_start to turn into FP64: the conversions
// (FP64 issue, 20 ns a step with one lane at work) are left to the block's
// other threads.  One warp's instruction stream bounds it (~110 per step): a
// step's drive terms are loaded during the step before.
// 25 600 steps: 2.08 ms; 2.88 with the conversions in it and one step a
// loop round.
template <int M, int FORCE>
__device__ __forceinline__ void guess_starts(const KAffine<float>& Kf, const Coef<float>& cf,
                                             const float* rows, int B, double* Y) {
    constexpr int S2 = 2 * M, W = aff::Rows<M, FORCE>::words;
    const aff::LawCoef<float> c = aff::law_coef(cf);
    aff::State<float, M, aff::MODE0> s;
    aff::init<float, M, aff::MODE0>(Kf, s);
    const float* row = rows;
    const float* end = rows + (size_t)(Kf.spc2 >> 1) * W;
    float R[W];
    aff::load_row<float, M, FORCE>(Kf, row, R);
    for (int b = 1; b < B; ++b) {   // (B - 1) AFM_SEG < n
#pragma unroll 2
        for (int k = 0; k < AFM_SEG; ++k) {
            row += W;
            if (row == end) row = rows;
            float Rn[W];
            aff::load_row<float, M, FORCE>(Kf, row, Rn);
            aff::step<float, M, FORCE, aff::MODE0>(Kf, c, R, s);
#pragma unroll
            for (int w = 0; w < W; ++w) R[w] = Rn[w];
        }
        float2* y = reinterpret_cast<float2*>(Y + (size_t)b * S2);
#pragma unroll
        for (int k = 0; k < M; ++k) {
            y[k] = make_float2(s.q[k], k == 0 ? s.cq[0] : 0.f);
            y[M + k] = make_float2(s.p[k], k == 0 ? s.cp[0] : 0.f);
        }
    }
}

// The start Y[2m] left by guess_starts as (deflections, rates) in FP64.
template <int M>
__device__ __forceinline__ void finish_start(const KAffine<double>& Kd, double* Y) {
    aff::State<float, M, aff::MODE0> s;
    const float2* y = reinterpret_cast<const float2*>(Y);
#pragma unroll
    for (int k = 0; k < M; ++k) {
        const float2 q = y[k], v = y[M + k];
        s.q[k] = q.x;
        s.p[k] = v.x;
        if (k == 0) {
            s.cq[0] = q.y;
            s.cp[0] = v.y;
        }
    }
    double q[M], v[M];
    aff::export_state<float, M, aff::MODE0>(Kd, s, q, v);
#pragma unroll
    for (int k = 0; k < M; ++k) {
        Y[k] = q[k];
        Y[M + k] = v[k];
    }
}

// Newton update of the segment starts, in order over the joins:
// Znew_0 = Zold_0 (the exact initial state), Znew_{b+1} = E_b + J_b (Znew_b -
// Zold_b); Znew may be Zold.  One warp, lanes i and 16 + i for component i:
// the even and the odd columns of the product.  Its chain bounds it: three
// FP64 products (for three modes), an addition and a subtraction at 64 clocks
// of issue each and two shuffles; the operands are loaded AHEAD joins before.
// 800 joins of three modes: 258 us, 510 with all columns in one lane and
// operands one join ahead.
template <int M, typename TJ>
__device__ __forceinline__ void correct_starts(const double* Zold, double* Znew, const double* E,
                                               const TJ* J, int B) {
    constexpr int S2 = 2 * M, AHEAD = 4;
    const int lane = threadIdx.x & 31, h = lane >> 4;
    const bool store = (lane & 15) < S2 && h == 0;
    const int i = (lane & 15) < S2 ? lane & 15 : 0;
    double z = Zold[i], e[AHEAD], y[AHEAD];
    // to FP64 one join ahead: at the load the conversion would wait for it, at
    // the use the chain for the conversion
    TJ Jr[AHEAD][M];
    double Jd[M];
    auto load = [&](int b, int k) {
        b = min(b, B - 1);
        const size_t o = (size_t)b * S2 + i;
        e[k] = E[o];
        y[k] = Zold[o];
#pragma unroll
        for (int c = 0; c < M; ++c) Jr[k][c] = J[o * S2 + 2 * c + h];
    };
    if (store) Znew[i] = z;
#pragma unroll
    for (int k = 0; k < AHEAD; ++k) load(k, k);
#pragma unroll
    for (int c = 0; c < M; ++c) Jd[c] = (double)Jr[0][c];
    for (int b0 = 0; b0 + 1 < B; b0 += AHEAD) {
#pragma unroll
        for (int k = 0; k < AHEAD; ++k) {
            const int b = b0 + k;
            if (b + 1 >= B) break;
            const double dl = z - y[k];
            double acc = h == 0 ? e[k] : 0.0;
#pragma unroll
            for (int c = 0; c < M; ++c)
                acc = fma(Jd[c], __shfl_sync(0xffffffffu, dl, 2 * c + h), acc);
#pragma unroll
            for (int c = 0; c < M; ++c) Jd[c] = (double)Jr[(k + 1) % AHEAD][c];
            load(b + AHEAD, k);   // reads starts that are replaced later
            z = acc + __shfl_xor_sync(0xffffffffu, acc, 16);
            if (store) Znew[(size_t)(b + 1) * S2 + i] = z;
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
