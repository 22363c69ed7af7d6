// kern_adjoint.cu -- discrete adjoint of the fused forward solve: gradient of
// the misfit S (Eq. 5) with respect to the normalised force parameters x,
// through every RK4 step of Eq. 2 (Sec. 3.2), one thread per particle.
//
// Forward pass: the RK4 loop of afm_device.cuh with every mode compensated
// (the gradient is more sensitive to the trajectory's rounding than the
// misfit; the forward kernels compensate the lowest mode only), storing the
// full state (modal deflections, rates and their Kahan compensations) every
// AFM_SEG steps.  Reverse pass: for each segment, last first, the AFM_SEG steps are
// recomputed from their checkpoint (bit-identical to the forward pass) while
// the gap d and gap rate d' of each RK4 stage and the tip deflection after
// each step are kept in shared memory; then the adjoint state runs back
// through the segment, one reverse RK4 step at a time, accumulating the
// cotangents of the four force coefficients.  A final chain rule maps them to
// d S / d x.
//
// One record for all particles and few particles (adj_split): such a launch
// takes one warp's chains, forward, recompute and reverse one after the other,
// ~520 ns a step in one kernel.  Only the forward solve is serial in time; the
// adjoint state is a linear recurrence, and its segments are run at once:
//   adj_forward_kernel   the solve with its checkpoints, in the affine form of
//                        the step (afm_affine.cuh)
//   adj_segment_kernel   (one thread per segment and particle) recomputes the
//                        steps and stores the force slopes of the four stages
//                        and the residual of each
//   adj_transfer_kernel  (one thread per segment, column and particle) the
//                        segment's map of the adjoint state, column by column,
//                        and its inhomogeneous part: the transposed affine
//                        step (afm_affine.cuh), ~110 operations
//   adj_join_kernel      the adjoint state at every segment's end, in FP64:
//                        one small matrix-vector product per segment
//   adj_segment_kernel   again: the adjoint state back through the segment,
//                        then the coefficients' cotangents
//   adj_final_kernel     their sums in FP64 and the chain rule
// The steepest-descent polish keeps the one kernel: a pixel polished alone
// takes the same bits as in a batch of ragged records.
// A column is a compensated FP32 recurrence (sum and compensation enter the
// map as one FP64 number), so a segment's rounding is that of the serial
// recurrence and the joins add none.  The affine form and the gaps' use of
// q_0's compensation halve the gradient's error against FP64 (2-norm over 32
// particles x 2560 steps, mean of 24 records: 6.3e-7 in one kernel, 3.5e-7).
// Measured (DMT, three modes, 32 particles x 2560 steps): 340 us, 1325 us in
// one kernel; 200 us of it the forward solve (78 ns a step), the chain left.
// With the adjoint state taken back serially, one lane a particle: 307 us for
// that pass alone.
#include <algorithm>
#include <type_traits>

#include "afm_affine.cuh"
#include "afm_device.cuh"
#include "afm_launch.h"
#include "afm_tangent.cuh"
#include "afm_warp.cuh"   // per_block

namespace afm {

constexpr int SEG = AFM_SEG;
constexpr int SEGW = 9;   // per step: (d, d') of 4 stages + tip deflection
constexpr int ADJ_THREADS = 32;

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

}  // namespace

// Transposed Jacobian of the modal right-hand side f(q, v) = (v, a) at one
// stage, applied to w = (wq, wv); accumulates the force-coefficient
// cotangents into cb.
template <int M, int FORCE>
__device__ __forceinline__ void rhs_vjp(const KConst<float>& K, const Coef<float>& c, float d,
                                        float dd, const float* wq, const float* wv, float* oq,
                                        float* ov, float* cb) {
    float Fd, Fr, Fc[4];
    force_partials<FORCE>(c, d, dd, Fd, Fr, Fc);
    float Fbar = 0.f;
#pragma unroll
    for (int i = 0; i < M; ++i) Fbar = fmaf(K.tip[i], wv[i], Fbar);
#pragma unroll
    for (int i = 0; i < M; ++i) {
        float aq = fmaf(Fbar, Fd, -K.w2[i] * wv[i]);
        if (i == 0) aq = fmaf(-K.w2lo[0], wv[0], aq);
        oq[i] = aq;
        ov[i] = wq[i] + fmaf(Fbar, Fr, -K.wq[i] * wv[i]);
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) cb[k] = fmaf(Fbar, Fc[k], cb[k]);
}

// One RK4 step as in rk4_step (every mode compensated), recording (d, d') of
// each stage.
template <int M, int FORCE>
__device__ __forceinline__ void rk4_step_rec(const KConst<float>& K, const Coef<float>& c, float* q,
                                             float* v, float* cq, float* cv, float g0, float gh,
                                             float g1, float* rec) {
    float a[M], qs[M], vs[M], Kq[M], Kv[M];
    auto gap = [&](const float* qq, const float* vv, int s) {
        float u = qq[0], r = vv[0];
#pragma unroll
        for (int i = 1; i < M; ++i) {
            u += qq[i];
            r += vv[i];
        }
        rec[2 * s] = K.Zc + u;
        rec[2 * s + 1] = r;
    };
    gap(q, v, 0);
    accel<float, M, FORCE>(K, c, q, v, g0, a);
#pragma unroll
    for (int i = 0; i < M; ++i) {
        Kq[i] = v[i];
        Kv[i] = a[i];
        qs[i] = fmaf(3.f, v[i], q[i]);
        vs[i] = fmaf(3.f, a[i], v[i]);
    }
    gap(qs, vs, 1);
    accel<float, M, FORCE>(K, c, qs, vs, gh, a);
#pragma unroll
    for (int i = 0; i < M; ++i) {
        Kq[i] = fmaf(2.f, vs[i], Kq[i]);
        Kv[i] = fmaf(2.f, a[i], Kv[i]);
        qs[i] = fmaf(3.f, vs[i], q[i]);
        vs[i] = fmaf(3.f, a[i], v[i]);
    }
    gap(qs, vs, 2);
    accel<float, M, FORCE>(K, c, qs, vs, gh, a);
#pragma unroll
    for (int i = 0; i < M; ++i) {
        Kq[i] = fmaf(2.f, vs[i], Kq[i]);
        Kv[i] = fmaf(2.f, a[i], Kv[i]);
        qs[i] = fmaf(6.f, vs[i], q[i]);
        vs[i] = fmaf(6.f, a[i], v[i]);
    }
    gap(qs, vs, 3);
    accel<float, M, FORCE>(K, c, qs, vs, g1, a);
#pragma unroll
    for (int i = 0; i < M; ++i) {
        Kq[i] = Kq[i] + vs[i];
        Kv[i] = Kv[i] + a[i];
        state_add<float, true>(i, q[i], cq[i], Kq[i]);
        state_add<float, true>(i, v[i], cv[i], Kv[i]);
    }
}

// (The pointer before the constants puts their arrays on 16-byte boundaries, see
// KConst: eight modes, 2048 particles x 5120 steps 4.70 ms, 4.75 eight bytes
// off.)
template <int M, int FORCE>
__global__ void __launch_bounds__(ADJ_THREADS) adjoint_kernel(const float* __restrict__ x,
                                                              const KConst<float> K, int P,
                                                              const float* __restrict__ U,
                                                              float* __restrict__ S_out,
                                                              float* __restrict__ G,
                                                              float* __restrict__ ckpt,
                                                              const int64_t* __restrict__ off,
                                                              const int* __restrict__ order,
                                                              int per_slot) {
    extern __shared__ __align__(16) float sma[];
    float* tab = sma;
    float* seg = sma + ((K.spc2 + 1 + 3) & ~3);   // [SEG][SEGW][ADJ_THREADS]
    build_drive_table(K, tab);
    __syncthreads();
    const int tid = threadIdx.x;
    const int p = blockIdx.x * blockDim.x + tid;
    if (p >= P) return;
    int N = K.n_steps;
    if (off != nullptr) {
        const int slot = p / per_slot;
        const int pix = order != nullptr ? order[slot] : slot;
        U += off[pix];
        N = (int)(off[pix + 1] - off[pix]);
        if (N > K.n_steps) {   // beyond the checkpoint buffer
            S_out[p] = INFINITY;
            for (int d = 0; d < K.D; ++d) G[(size_t)d * P + p] = 0.f;
            return;
        }
    }
    const int nseg = (N + SEG - 1) / SEG;
    float xd[AFM_MAXD];
    for (int d = 0; d < K.D; ++d) xd[d] = x[(size_t)d * P + p];
    const Coef<float> c = make_coef<float, float>(K, xd);

    // forward pass with checkpoints
    float q[M], v[M], cq[M], cv[M];
    init_state<float, M>(K, q, v, cq, cv);
    float S = 0.f, cS = 0.f;
    int j = 0;
    for (int n = 0; n < N; ++n) {
        if (n % SEG == 0) {
            float* ck = ckpt + (size_t)(n / SEG) * 4 * M * P + p;
#pragma unroll
            for (int i = 0; i < M; ++i) {
                ck[(size_t)(0 * M + i) * P] = q[i];
                ck[(size_t)(1 * M + i) * P] = v[i];
                ck[(size_t)(2 * M + i) * P] = cq[i];
                ck[(size_t)(3 * M + i) * P] = cv[i];
            }
        }
        const float g0 = tab[j], gh = tab[j + 1], g1 = tab[j + 2];
        j += 2;
        if (j >= K.spc2) j = 0;
        rk4_step<float, M, FORCE, true>(K, c, q, v, cq, cv, g0, gh, g1);
        const float r = U[n] - tip_sum<float, M>(q);
        const float y = fmaf(r, r, -cS);
        const float t = add_rn(S, y);
        cS = sub_rn(sub_rn(t, S), y);
        S = t;
    }
    S_out[p] = S;

    // reverse pass
    // adjoint state with Kahan compensations: like the forward state it takes
    // per-step increments far smaller than itself over the whole record
    float lq[M], lv[M], clq[M], clv[M];
#pragma unroll
    for (int i = 0; i < M; ++i) lq[i] = lv[i] = clq[i] = clv[i] = 0.f;
    // force-coefficient cotangents: FP32 within a segment, folded into FP64
    // after each (the sum runs over every stage of every step)
    double cbd[4] = {0.0, 0.0, 0.0, 0.0};
    for (int sg = nseg - 1; sg >= 0; --sg) {
        float cb[4] = {0.f, 0.f, 0.f, 0.f};
        const int n0 = sg * SEG, n1 = min(N, n0 + SEG);
        const float* ck = ckpt + (size_t)sg * 4 * M * P + p;
#pragma unroll
        for (int i = 0; i < M; ++i) {
            q[i] = ck[(size_t)(0 * M + i) * P];
            v[i] = ck[(size_t)(1 * M + i) * P];
            cq[i] = ck[(size_t)(2 * M + i) * P];
            cv[i] = ck[(size_t)(3 * M + i) * P];
        }
        int jj = (int)(((long long)2 * n0) % K.spc2);
        for (int n = n0; n < n1; ++n) {
            const float g0 = tab[jj], gh = tab[jj + 1], g1 = tab[jj + 2];
            jj += 2;
            if (jj >= K.spc2) jj = 0;
            float rec[8];
            rk4_step_rec<M, FORCE>(K, c, q, v, cq, cv, g0, gh, g1, rec);
            float* sb = seg + (size_t)(n - n0) * SEGW * ADJ_THREADS + tid;
#pragma unroll
            for (int k = 0; k < 8; ++k) sb[k * ADJ_THREADS] = rec[k];
            sb[8 * ADJ_THREADS] = tip_sum<float, M>(q);
        }
        for (int n = n1 - 1; n >= n0; --n) {
            const float* sb = seg + (size_t)(n - n0) * SEGW * ADJ_THREADS + tid;
            // misfit term of the state after step n
            const float r = U[n] - sb[8 * ADJ_THREADS];
#pragma unroll
            for (int i = 0; i < M; ++i) kahan_add(lq[i], clq[i], -2.f * r);
            // reverse RK4 step: stage cotangents kb_s (k1..k4 weights 1,2,2,1)
            float k1q[M], k1v[M], k2q[M], k2v[M], k3q[M], k3v[M], oq[M], ov[M];
            float yq[M], yv[M];
#pragma unroll
            for (int i = 0; i < M; ++i) {
                yq[i] = 0.f;   // the step's increment of the adjoint state
                yv[i] = 0.f;
                k1q[i] = lq[i];
                k1v[i] = lv[i];
                k2q[i] = 2.f * lq[i];
                k2v[i] = 2.f * lv[i];
                k3q[i] = 2.f * lq[i];
                k3v[i] = 2.f * lv[i];
            }
            // stage 4 (y4 = y + 6 k3), weight 1
            rhs_vjp<M, FORCE>(K, c, sb[6 * ADJ_THREADS], sb[7 * ADJ_THREADS], lq, lv, oq, ov, cb);
#pragma unroll
            for (int i = 0; i < M; ++i) {
                yq[i] += oq[i];
                yv[i] += ov[i];
                k3q[i] = fmaf(6.f, oq[i], k3q[i]);
                k3v[i] = fmaf(6.f, ov[i], k3v[i]);
            }
            // stage 3 (y3 = y + 3 k2)
            rhs_vjp<M, FORCE>(K, c, sb[4 * ADJ_THREADS], sb[5 * ADJ_THREADS], k3q, k3v, oq, ov, cb);
#pragma unroll
            for (int i = 0; i < M; ++i) {
                yq[i] += oq[i];
                yv[i] += ov[i];
                k2q[i] = fmaf(3.f, oq[i], k2q[i]);
                k2v[i] = fmaf(3.f, ov[i], k2v[i]);
            }
            // stage 2 (y2 = y + 3 k1)
            rhs_vjp<M, FORCE>(K, c, sb[2 * ADJ_THREADS], sb[3 * ADJ_THREADS], k2q, k2v, oq, ov, cb);
#pragma unroll
            for (int i = 0; i < M; ++i) {
                yq[i] += oq[i];
                yv[i] += ov[i];
                k1q[i] = fmaf(3.f, oq[i], k1q[i]);
                k1v[i] = fmaf(3.f, ov[i], k1v[i]);
            }
            // stage 1 (y)
            rhs_vjp<M, FORCE>(K, c, sb[0], sb[1 * ADJ_THREADS], k1q, k1v, oq, ov, cb);
#pragma unroll
            for (int i = 0; i < M; ++i) {
                kahan_add(lq[i], clq[i], yq[i] + oq[i]);
                kahan_add(lv[i], clv[i], yv[i] + ov[i]);
            }
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) cbd[k] += (double)cb[k];
    }
    double J[4][AFM_MAXD];
    coef_jacobian<float>(K, xd, J);
    for (int d = 0; d < K.D; ++d) {
        double g = 0.0;
        for (int k = 0; k < 4; ++k) g += cbd[k] * J[k][d];
        G[(size_t)d * P + p] = (float)g;
    }
}

// ---------------------------------------------------------------------------
// Few particles on one record.
// ---------------------------------------------------------------------------
namespace {

// The records of a launch behind its checkpoints.  T: the segments' maps,
// [segment][particle][row][2 M columns and the inhomogeneous part], then the
// adjoint state at the segments' ends in T's place: row i's in its first word
// (float2: value, compensation).  f: the stage force slopes by the gap
// [step][P], later the stage force cotangents in their place; g: the slopes by
// its rate (rate laws); cb: the coefficients' cotangents [segment][P]; r: the
// residuals [step][P].
struct Recs {
    double* T;
    float4 *f, *g, *cb;
    float* r;
};

__host__ __device__ constexpr int map_words(int M) { return 2 * M * (2 * M + 1); }
int tmodes(int m) { return m == 1 ? 1 : (m == 3 ? 3 : AFM_MAXM); }   // dispatch_mf's

size_t split_floats(int M, bool rate, int n_steps, int P) {
    const size_t seg = (size_t)((n_steps + SEG - 1) / SEG);
    return ((rate ? 9 : 5) * (size_t)n_steps + (4 + 2 * map_words(M)) * seg) * P;
}

// Where the split form pays.  It saves ~0.4 us of one warp's serial time a
// step, and costs five more launches (~55 us) and the work of the maps' 2 M + 1
// columns and the way back, ~0.05 ns x P a step and column, which the one
// kernel's idle SMs would not have done.  Measured, one kernel / split:
//   few particles (32): 128 steps 0.8 (1 mode) .. 1.15 (8), 160 0.96 .. 1.27,
//     200 1.08 .. 1.45, 256 1.2 .. 1.6, 512 1.7 .. 2.4, 2500 3.1 .. 4.0
//   break-even particles at 200 / 256 / 512 / 1000 steps: 1 mode (DMT) 700 /
//     1600 / 3800 / 5800; 3 modes (DMT and DMT + KV) 2000 / 2300 / 3700 / 5000,
//     (spring-damper) 4000 at 1000; 8 modes (Hooke) past 2222 from 256 on,
//     (spring-damper) 1450 / 1800 / 2100 / 2300
//   its blocks build their drive rows, which shows past 512 phases: at 1280
//     steps 3 modes break even at 4000 particles with 1024 phases and 2700 with
//     2048, 8 modes (spring-damper) past 1700 and at 1400
// The lines below stay within those (0.97 at their worst).
long long split_max_particles(int M, int force, int n_steps) {
    const long long n = n_steps;
    const bool rate = rate_law(force), kv = force == F_DMT_KV;
    long long most, rise, flat = 2000 + 12 * n / 5;
    if (M == 1) {   // DMT + KV: the one kernel's step is 1.3 times DMT's
        most = rate && !kv ? 4500 : 6000;
        rise = kv ? 20 * (n - 150) : 12 * (n - (rate ? 155 : 170));
        if (kv) flat = 2500 + 3 * n;
    } else if (M == 3) {
        most = rate ? 4000 : 5000;
        rise = rate ? 18 * (n - 140) : 17 * (n - 130);
    } else {
        most = rate ? 1500 + n / 2 : 2222;
        rise = rate ? 13 * (n - 130) : 15 * (n - 110);
    }
    return std::max(0ll, std::min({most, rise, flat}));
}

// Its records stay within 256 MB.
constexpr size_t SPLIT_FLOATS = 64u << 20;

bool adj_split(int M, int force, int n_steps, int spc, int P) {
    return P <= split_max_particles(M, force, n_steps) && (long long)P * spc <= (M <= 3 ? 4000000 : 1500000) &&
           split_floats(M, rate_law(force), n_steps, P) <= SPLIT_FLOATS;
}

// One step of the adjoint state back in time: the cotangents lq, lp of the
// state (q, second coordinate) after the step, compensated, to those before
// it; r2: the misfit term of the state after the step; Fd, Fr: the slopes of
// the stage forces; F: their cotangents.
template <int M, int FORCE>
__device__ __forceinline__ void reverse_step(const Affine<float>& A, const float* Fd,
                                             const float* Fr, float r2, float* lq, float* clq,
                                             float* lp, float* clp, float* F) {
    constexpr bool rate = UsesRate<FORCE>::value;
    // cotangents of the state after the step with its misfit term, then of
    // the stage forces, last stage first
    float l[M], d[4], r[4];
#pragma unroll
    for (int i = 0; i < M; ++i) l[i] = lq[i] + r2;
#pragma unroll
    for (int s = 0; s < 4; ++s) {
        float a = A.bp[s][0] * lp[0], b = 0.f;
        if (s < 3) b = A.bq[s][0] * l[0];
#pragma unroll
        for (int i = 1; i < M; ++i) {
            a = fmaf(A.bp[s][i], lp[i], a);
            if (s < 3) b = fmaf(A.bq[s][i], l[i], b);
        }
        F[s] = s < 3 ? a + b : a;
        r[s] = 0.f;
    }
    d[3] = Fd[3] * F[3];
    if constexpr (rate) {
        r[3] = Fr[3] * F[3];
        F[2] = fmaf(A.h43, r[3], F[2]);
    }
    d[2] = Fd[2] * F[2];
    F[1] = fmaf(A.e42, d[3], F[1]);
    if constexpr (rate) {
        r[2] = Fr[2] * F[2];
        F[1] = fmaf(A.h42, r[3], fmaf(A.h32, r[2], F[1]));
    }
    d[1] = Fd[1] * F[1];
    F[0] = fmaf(A.e41, d[3], fmaf(A.e31, d[2], F[0]));
    if constexpr (rate) {
        r[1] = Fr[1] * F[1];
        F[0] = fmaf(A.h41, r[3], fmaf(A.h31, r[2], fmaf(A.h21, r[1], F[0])));
    }
    d[0] = Fd[0] * F[0];
    if constexpr (rate) r[0] = Fr[0] * F[0];
    // increments of the state's cotangents, small terms first
    float iq[M], ip[M];
    iq[0] = A.d2q * d[1];
    ip[0] = A.d2w * d[1];
#pragma unroll
    for (int i = 0; i < M; ++i) {
        if (i > 0) {
            iq[i] = d[0] + d[1];
            ip[i] = d[1];
        }
        iq[i] = fmaf(A.d3q[i], d[2], fmaf(A.d4q[i], d[3], iq[i]));
        ip[i] = fmaf(A.d3p[i], d[2], fmaf(A.d4p[i], d[3], ip[i]));
        if constexpr (rate) {
            iq[i] = fmaf(A.r2q[i], r[1], fmaf(A.r3q[i], r[2], fmaf(A.r4q[i], r[3], iq[i])));
            ip[i] = fmaf(A.r2p[i], r[1], fmaf(A.r3p[i], r[2], fmaf(A.r4p[i], r[3], ip[i])));
            if (i > 0)
                ip[i] = fmaf(A.third, r[0], ip[i]);
            else {
                iq[i] = fmaf(A.v1q, r[0], iq[i]);
                ip[i] = fmaf(A.v1w, r[0], ip[i]);
            }
        }
    }
    iq[0] = fmaf(A.c0lo, lp[0], iq[0]) + ((d[0] + d[1]) + (d[2] + d[3]));
    ip[0] = fmaf(A.ec, lp[0], fmaf(A.c0lo, lp[0], ip[0]));
    iq[0] = fmaf(A.c0, lp[0], iq[0]);
    ip[0] = fmaf(A.c0, lp[0], ip[0]) + l[0];
#pragma unroll
    for (int i = 1; i < M; ++i) {
        iq[i] = fmaf(A.A1[i], l[i], fmaf(A.C[i], lp[i], iq[i]));
        ip[i] = fmaf(A.D1[i], lp[i], fmaf(A.B[i], l[i], ip[i]));
    }
#pragma unroll
    for (int i = 0; i < M; ++i) {
        kahan_add(lq[i], clq[i], r2 + iq[i]);
        kahan_add(lp[i], clp[i], ip[i]);
    }
}

}  // namespace

// The solve with a checkpoint before every SEG steps, one lane per particle:
// record values read 32 at a time and handed out by shuffles, a step's drive
// terms loaded during the step before (afm_warp.cuh).
template <int M, int FORCE>
__global__ void __launch_bounds__(128, 1)
adj_forward_kernel(const KAffine<float> K, const float* __restrict__ x, int P, int ppb,
                   const float* __restrict__ U, float* __restrict__ S_out,
                   float* __restrict__ ckpt) {
    constexpr int W = aff::Rows<M, FORCE>::words;
    extern __shared__ __align__(16) float sma[];
    aff::build_rows<float, M, FORCE>(K, sma);
    __syncthreads();
    const int p0 = blockIdx.x * ppb + threadIdx.x;
    if ((int)(threadIdx.x & ~31u) >= ppb || (p0 & ~31) >= P) return;   // whole warps
    const bool store = p0 < P;
    const int p = min(p0, P - 1), lane = threadIdx.x & 31, n = K.n_steps;
    float xd[AFM_MAXD];
    for (int d = 0; d < K.D; ++d) xd[d] = x[(size_t)d * P + p];
    const aff::LawCoef<float> c = aff::law_coef(make_coef<float, float>(K, xd));
    aff::State<float, M, aff::ALL> s;
    aff::init<float, M, aff::ALL>(K, s);
    float S = 0.f, cS = 0.f, R[W];
    const float* row = sma;
    const float* end = sma + (size_t)(K.spc2 >> 1) * W;
    aff::load_row<float, M, FORCE>(K, row, R);
    float Ub = lane < n ? U[lane] : 0.f;
    auto one = [&](int k) {
        row += W;
        if (row == end) row = sma;
        float Rn[W];
        aff::load_row<float, M, FORCE>(K, row, Rn);
        const float Un = __shfl_sync(0xffffffffu, Ub, k);
        aff::step<float, M, FORCE, aff::ALL>(K, c, R, s);
        aff::misfit_add(Un, aff::tip<float, M, aff::ALL>(s), S, cS);
#pragma unroll
        for (int w = 0; w < W; ++w) R[w] = Rn[w];
    };
    static_assert(SEG == 32, "a checkpoint per block of record values");
    for (int k0 = 0; k0 < n; k0 += SEG) {
        if (store) {
            float* ck = ckpt + (size_t)(k0 / SEG) * 4 * M * P + p;
#pragma unroll
            for (int i = 0; i < M; ++i) {
                ck[(size_t)(0 * M + i) * P] = s.q[i];
                ck[(size_t)(1 * M + i) * P] = s.p[i];
                ck[(size_t)(2 * M + i) * P] = s.cq[i];
                ck[(size_t)(3 * M + i) * P] = s.cp[i];
            }
        }
        const int kn = k0 + SEG + lane;
        const float Unb = kn < n ? U[kn] : 0.f;
        if (k0 + SEG <= n) {
#pragma unroll 2
            for (int k = 0; k < SEG; ++k) one(k);
        } else {
            for (int k = 0; k < n - k0; ++k) one(k);
        }
        Ub = Unb;
    }
    if (store) S_out[p] = S;
}

// COEF = false: slopes and residuals of every step.  true: the adjoint state
// back through the segment, leaving the stage force cotangents, then the
// segment's sums of the coefficients' cotangents.
template <int M, int FORCE, bool COEF>
__global__ void __launch_bounds__(128)
adj_segment_kernel(const KAffine<float> K, const float* __restrict__ x, int P, int nseg,
                   const float* __restrict__ U, const float* __restrict__ ckpt, const Recs R) {
    constexpr int NC = aff::CoefDirs<FORCE>::n;
    constexpr int W = aff::Rows<M, FORCE>::words;
    extern __shared__ __align__(16) float sma[];
    aff::build_rows<float, M, FORCE>(K, sma);
    __syncthreads();
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= (long long)nseg * P) return;
    const int sg = (int)(t / P), p = (int)(t % P);
    const int n0 = sg * SEG, n1 = min(K.n_steps, n0 + SEG);
    if constexpr (COEF) {
        float lq[M], lp[M], clq[M], clp[M], F[4];
        const double* T = R.T + ((size_t)sg * P + p) * map_words(M);
#pragma unroll
        for (int i = 0; i < M; ++i) {
            const float2 a = *reinterpret_cast<const float2*>(T + i * (2 * M + 1));
            const float2 b = *reinterpret_cast<const float2*>(T + (M + i) * (2 * M + 1));
            lq[i] = a.x;
            clq[i] = a.y;
            lp[i] = b.x;
            clp[i] = b.y;
        }
        float4 fn = R.f[(size_t)(n1 - 1) * P + p], gn = fn;
        if constexpr (UsesRate<FORCE>::value) gn = R.g[(size_t)(n1 - 1) * P + p];
        float rn = R.r[(size_t)(n1 - 1) * P + p];
        for (int n = n1 - 1; n >= n0; --n) {
            const float Fd[4] = {fn.x, fn.y, fn.z, fn.w}, Fr[4] = {gn.x, gn.y, gn.z, gn.w};
            const float r2 = -2.f * rn;
            if (n > n0) {   // a step ahead
                fn = R.f[(size_t)(n - 1) * P + p];
                if constexpr (UsesRate<FORCE>::value) gn = R.g[(size_t)(n - 1) * P + p];
                rn = R.r[(size_t)(n - 1) * P + p];
            }
            reverse_step<M, FORCE>(K.af, Fd, Fr, r2, lq, clq, lp, clp, F);
            R.f[(size_t)n * P + p] = make_float4(F[0], F[1], F[2], F[3]);
        }
    }
    float xd[AFM_MAXD];
    for (int d = 0; d < K.D; ++d) xd[d] = x[(size_t)d * P + p];
    const Coef<float> c = make_coef<float, float>(K, xd);
    const aff::LawCoef<float> lc = aff::law_coef(c);
    aff::State<float, M, aff::ALL> s;
    const float* ck = ckpt + (size_t)sg * 4 * M * P + p;
#pragma unroll
    for (int i = 0; i < M; ++i) {
        s.q[i] = ck[(size_t)(0 * M + i) * P];
        s.p[i] = ck[(size_t)(1 * M + i) * P];
        s.cq[i] = ck[(size_t)(2 * M + i) * P];
        s.cp[i] = ck[(size_t)(3 * M + i) * P];
    }
    s.s1 = aff::sum_tail<float, M>(s.q);
    const int spc = K.spc2 >> 1;
    int j = n0 % spc;
    float cb[NC], ccb[NC];
#pragma unroll
    for (int k = 0; k < NC; ++k) cb[k] = ccb[k] = 0.f;
    float4 Fn = make_float4(0.f, 0.f, 0.f, 0.f);   // next step's cotangents
    if constexpr (COEF) Fn = R.f[(size_t)n0 * P + p];
    for (int n = n0; n < n1; ++n) {
        float Rw[W];
        aff::load_row<float, M, FORCE>(K, sma + (size_t)j * W, Rw);
        if (++j == spc) j = 0;
        const float Fb[4] = {Fn.x, Fn.y, Fn.z, Fn.w};
        if constexpr (COEF) {
            if (n + 1 < n1) Fn = R.f[(size_t)(n + 1) * P + p];
        }
        aff::Stages<float> g;
        aff::stages<float, M, FORCE, aff::ALL>(K, lc, Rw, s, g);
        aff::advance<float, M, aff::ALL>(K, Rw, g.F, s);
        float Fd[4], Fr[4], sum[NC];
#pragma unroll
        for (int l = 0; l < NC; ++l) sum[l] = 0.f;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            aff::Partials<FORCE> Ps;
            aff::partials<FORCE>(c, g.d[k], g.r[k], Ps);
            Fd[k] = Ps.Fd;
            Fr[k] = Ps.Fr;
            if constexpr (COEF) {
#pragma unroll
                for (int l = 0; l < NC; ++l) sum[l] = fmaf(Fb[k], Ps.Fc[l], sum[l]);
            }
        }
        if constexpr (COEF) {
#pragma unroll
            for (int l = 0; l < NC; ++l) kahan_add(cb[l], ccb[l], sum[l]);
        }
        if constexpr (!COEF) {
            R.f[(size_t)n * P + p] = make_float4(Fd[0], Fd[1], Fd[2], Fd[3]);
            if constexpr (UsesRate<FORCE>::value)
                R.g[(size_t)n * P + p] = make_float4(Fr[0], Fr[1], Fr[2], Fr[3]);
            // with the compensations: the deflection's own rounding is a
            // visible part of a small residual
            const float e = __fsub_rn(U[n], s.q[0]);
            float rest = s.cq[0];
#pragma unroll
            for (int i = 1; i < M; ++i) rest += s.cq[i] - s.q[i];
            R.r[(size_t)n * P + p] = __fadd_rn(e, rest);
        }
    }
    if constexpr (COEF) {
        float o[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int l = 0; l < NC; ++l) o[aff::CoefDirs<FORCE>::index(l)] = cb[l];
        R.cb[(size_t)sg * P + p] = make_float4(o[0], o[1], o[2], o[3]);
    }
}

// The segments' maps: column c < 2 M of the transposed step's product, or
// (c = 2 M) the adjoint state that the segment's residuals give from zero.
template <int M, int FORCE>
__global__ void __launch_bounds__(128)
adj_transfer_kernel(const KAffine<float> K, int P, int nseg, const Recs R) {
    constexpr int D2 = 2 * M, W = D2 + 1;
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= (long long)nseg * P * W) return;
    const int p = (int)(t % P), c = (int)(t / P % W), sg = (int)(t / P / W);
    const int n0 = sg * SEG, n1 = min(K.n_steps, n0 + SEG);
    float lq[M], lp[M], clq[M], clp[M], F[4];
#pragma unroll
    for (int i = 0; i < M; ++i) {
        lq[i] = c == i ? 1.f : 0.f;
        lp[i] = c == M + i ? 1.f : 0.f;
        clq[i] = clp[i] = 0.f;
    }
    const float rs = c == D2 ? -2.f : 0.f;
    float4 fn = R.f[(size_t)(n1 - 1) * P + p], gn = fn;
    if constexpr (UsesRate<FORCE>::value) gn = R.g[(size_t)(n1 - 1) * P + p];
    float rn = R.r[(size_t)(n1 - 1) * P + p];
    for (int n = n1 - 1; n >= n0; --n) {
        const float Fd[4] = {fn.x, fn.y, fn.z, fn.w}, Fr[4] = {gn.x, gn.y, gn.z, gn.w};
        const float r2 = rs == 0.f ? 0.f : rs * rn;
        if (n > n0) {   // a step ahead
            fn = R.f[(size_t)(n - 1) * P + p];
            if constexpr (UsesRate<FORCE>::value) gn = R.g[(size_t)(n - 1) * P + p];
            rn = R.r[(size_t)(n - 1) * P + p];
        }
        reverse_step<M, FORCE>(K.af, Fd, Fr, r2, lq, clq, lp, clp, F);
    }
    double* o = R.T + ((size_t)sg * P + p) * map_words(M) + c;
#pragma unroll
    for (int i = 0; i < M; ++i) {
        o[i * W] = (double)lq[i] - (double)clq[i];
        o[(M + i) * W] = (double)lp[i] - (double)clp[i];
    }
}

// The adjoint state at the end of every segment, last first; one lane per
// particle and row (ROWS: 2 M rounded up to a power of two).
template <int M, int ROWS>
__global__ void __launch_bounds__(32)
adj_join_kernel(int P, int nseg, const Recs R) {
    constexpr int D2 = 2 * M, W = D2 + 1;
    const int per = 32 / ROWS, lane = threadIdx.x, base = lane & ~(ROWS - 1);
    const int p = min(P - 1, (int)blockIdx.x * per + lane / ROWS);
    const int row = min(lane % ROWS, D2 - 1);
    const bool store = (int)blockIdx.x * per + lane / ROWS < P && lane % ROWS < D2;
    const size_t stride = (size_t)P * map_words(M);
    double* T = R.T + (size_t)p * map_words(M) + (size_t)row * W;
    // rows of the next AHEAD segments in registers (a load takes longer than a
    // segment's product)
    constexpr int AHEAD = 4;
    double a[AHEAD][W];
    auto load = [&](int sg, double* v) {
        if (sg >= 0) {
#pragma unroll
            for (int k = 0; k < W; ++k) v[k] = T[sg * stride + k];
        }
    };
#pragma unroll
    for (int k = 0; k < AHEAD; ++k) load(nseg - 1 - k, a[k]);
    double l = 0.0;
    auto one = [&](int sg, double* v) {
        double s = v[D2], s2 = 0.0;
        if (sg < nseg - 1) {
#pragma unroll
            for (int k = 0; k < D2; k += 2) {
                s = fma(v[k], __shfl_sync(0xffffffffu, l, base + k), s);
                s2 = fma(v[k + 1], __shfl_sync(0xffffffffu, l, base + k + 1), s2);
            }
        }
        __syncwarp();
        load(sg - AHEAD, v);
        // the state at this segment's end; every lane has read its row
        if (store) {
            const float hi = (float)l;
            *reinterpret_cast<float2*>(T + sg * stride) = make_float2(hi, (float)((double)hi - l));
        }
        l = s + s2;
    };
    for (int sg = nseg - 1; sg >= 0; sg -= AHEAD) {
#pragma unroll
        for (int k = 0; k < AHEAD; ++k)
            if (k <= sg) one(sg - k, a[k]);
    }
}

// G = J^T (sums over the segments), one warp per particle.
__global__ void __launch_bounds__(128)
adj_final_kernel(const KConst<float> K, const float* __restrict__ x, int P, int nseg,
                 const float4* __restrict__ cbs, float* __restrict__ G) {
    const int p = (int)((blockIdx.x * (size_t)blockDim.x + threadIdx.x) >> 5);
    const int lane = threadIdx.x & 31;
    if (p >= P) return;
    double cb[4] = {0.0, 0.0, 0.0, 0.0};
    for (int sg = lane; sg < nseg; sg += 32) {
        const float4 v = cbs[(size_t)sg * P + p];
        cb[0] += (double)v.x;
        cb[1] += (double)v.y;
        cb[2] += (double)v.z;
        cb[3] += (double)v.w;
    }
#pragma unroll
    for (int k = 0; k < 4; ++k)
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) cb[k] += __shfl_xor_sync(0xffffffffu, cb[k], o);
    if (lane != 0) return;
    float xd[AFM_MAXD];
    for (int d = 0; d < K.D; ++d) xd[d] = x[(size_t)d * P + p];
    double J[4][AFM_MAXD];
    coef_jacobian<float>(K, xd, J);
    for (int d = 0; d < K.D; ++d) {
        double g = 0.0;
        for (int k = 0; k < 4; ++k) g += cb[k] * J[k][d];
        G[(size_t)d * P + p] = (float)g;
    }
}

// The checkpoints, 16 byte multiples.
size_t adjoint_ckpt_floats(int m, int n_steps, int P) {
    return (size_t)((n_steps + SEG - 1) / SEG) * 4 * tmodes(m) * P;
}

// The checkpoints with room for the split form's records at P particles and
// below: it grows with P and with n_steps, so a buffer of a larger batch's or a
// longer record's size serves a smaller one's split form too.
size_t adjoint_ws_floats(int m, int force, int n_steps, int P) {
    const int M = tmodes(m);
    const int Ps = (int)std::min((long long)P, split_max_particles(M, force, n_steps));
    const size_t split = adjoint_ckpt_floats(m, n_steps, Ps) +
                         std::min(split_floats(M, rate_law(force), n_steps, Ps), SPLIT_FLOATS);
    return std::max(adjoint_ckpt_floats(m, n_steps, P), split);
}

bool adjoint_runs_split(int m, int force, int n_steps, int spc, int P, const void* ws,
                        size_t ws_bytes) {
    const int M = tmodes(m);
    return adj_split(M, force, n_steps, spc, P) && reinterpret_cast<uintptr_t>(ws) % 16 == 0 &&
           ws_bytes / sizeof(float) >= adjoint_ckpt_floats(m, n_steps, P) +
                                           split_floats(M, rate_law(force), n_steps, P);
}

cudaError_t launch_adjoint_split(const KAffine<float>& K, const float* x, int P, const float* U,
                                 float* S, float* G, float* ckpt, cudaStream_t st) {
    const int nseg = (K.n_steps + SEG - 1) / SEG;
    const int ppb = warp::per_block(P), blocks = (P + ppb - 1) / ppb;
    auto per128 = [](long long n) { return (int)((n + 127) / 128); };
    return dispatch_mf(K.m, K.force, [&](auto Mc, auto Fc) -> cudaError_t {
        constexpr int M = decltype(Mc)::value, FORCE = decltype(Fc)::value;
        constexpr int ROWS = M == 1 ? 2 : (M == 3 ? 8 : 2 * AFM_MAXM);
        Recs R;
        R.f = reinterpret_cast<float4*>(ckpt + adjoint_ckpt_floats(K.m, K.n_steps, P));
        R.g = R.f + (size_t)K.n_steps * P;
        R.cb = UsesRate<FORCE>::value ? R.g + (size_t)K.n_steps * P : R.g;
        R.T = reinterpret_cast<double*>(R.cb + (size_t)nseg * P);
        R.r = reinterpret_cast<float*>(R.T + (size_t)nseg * P * map_words(M));
        const int sblocks = per128((long long)nseg * P);
        const size_t smem = aff_table_bytes<float, M, FORCE>(K.spc2);
        if (smem > 48 * 1024) {
            auto large = [&](auto k) {
                return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
            };
            cudaError_t e = large(adj_forward_kernel<M, FORCE>);
            if (e == cudaSuccess) e = large(adj_segment_kernel<M, FORCE, false>);
            if (e == cudaSuccess) e = large(adj_segment_kernel<M, FORCE, true>);
            if (e != cudaSuccess) return e;
        }
        adj_forward_kernel<M, FORCE><<<blocks, 128, smem, st>>>(K, x, P, ppb, U, S, ckpt);
        adj_segment_kernel<M, FORCE, false><<<sblocks, 128, smem, st>>>(K, x, P, nseg, U, ckpt, R);
        adj_transfer_kernel<M, FORCE><<<per128((long long)nseg * P * (2 * M + 1)), 128, 0, st>>>(
            K, P, nseg, R);
        adj_join_kernel<M, ROWS><<<(P + 32 / ROWS - 1) / (32 / ROWS), 32, 0, st>>>(P, nseg, R);
        adj_segment_kernel<M, FORCE, true><<<sblocks, 128, smem, st>>>(K, x, P, nseg, U, ckpt, R);
        adj_final_kernel<<<per128(32ll * P), 128, 0, st>>>(K, x, P, nseg, R.cb, G);
        return cudaGetLastError();
    });
}

cudaError_t launch_adjoint(const KConst<float>& K, const float* x, int P, const float* U, float* S,
                           float* G, float* ckpt, cudaStream_t st, const int64_t* off,
                           const int* order, int per_slot) {
    const size_t smem = sizeof(float) * ((size_t)((K.spc2 + 1 + 3) & ~3) +
                                         (size_t)SEG * SEGW * ADJ_THREADS);
    const int blocks = (P + ADJ_THREADS - 1) / ADJ_THREADS;
    return dispatch_mf(K.m, K.force, [&](auto Mc, auto Fc) -> cudaError_t {
        auto kern = adjoint_kernel<decltype(Mc)::value, decltype(Fc)::value>;
        if (smem > 48 * 1024) {
            cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                 (int)smem);
            if (e != cudaSuccess) return e;
        }
        kern<<<blocks, ADJ_THREADS, smem, st>>>(x, K, P, U, S, G, ckpt, off, order, per_slot);
        return cudaGetLastError();
    });
}

}  // namespace afm
