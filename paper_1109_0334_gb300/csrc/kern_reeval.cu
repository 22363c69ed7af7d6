// kern_reeval.cu -- FP64 re-evaluation of one winner's misfit (Eq. 5 on the
// RK4 solution of Eq. 2, Sec. 3.2) by multiple shooting in time.
//
// FP64 arithmetic on this GPU issues at a small fraction of the FP32 rate,
// so one thread stepping a whole record in FP64 needs 5 to 7 us per RK4 step.
// The record is instead cut into segments of AFM_SEG steps that are
// integrated concurrently, one thread each, and the segment start states
// are made consistent by Newton's method on the matching conditions
// Z_{b+1} = Phi_b(Z_b), Phi_b being AFM_SEG FP64 RK4 steps:
//   guess  one thread integrates the winner in FP32 (compensated, in the
//          affine form) and keeps the state at every segment start;
//   sweep  (twice) every segment is integrated in FP64 from its start Z_b,
//          giving E_b = Phi_b(Z_b), while its tangent map J_b = dPhi_b/dZ_b
//          is propagated in FP32 (the RK4 step linearised about the FP64
//          stages); one warp then walks the joins in order:
//          Z'_0 = y_0,  Z'_{b+1} = E_b + J_b (Z'_b - Z_b);
//   final  the segments are integrated in FP64 from the corrected starts,
//          each summing its share of the misfit; S is the FP64 sum of the
//          shares.
// The joins are then checked: if the summed max-norm mismatch between each
// segment's end and the next segment's start exceeds 1e-9 (scaled units),
// or anything is non-finite, the final kernel integrates the whole record
// once more, sequentially, in FP64.
//
// A 25 600-step record (three modes, DMT): guess 2.08 ms (one thread's
// 25 600 FP32 steps, most of what is left), three passes 0.58 ms, two walks
// over the joins 0.52 ms; with the stage form, conversions in the guess and
// all columns of a join in one lane ~6 ms.
#include "afm_reeval.cuh"

namespace afm {

using namespace reeval;

// The swarm's global best (as invert_final_kernel selects it); one thread.
__global__ void reeval_pick_swarm_kernel(const PsoConst pc, const SwarmPtrs sw, float* history,
                                         ReevalWinner* __restrict__ w) {
    const int fin = (pc.iters + 1) & 1;
    const unsigned long long key = *sw.gkey[fin];
    const int g = min((int)(key & 0x7fffffffu), pc.P - 1);
    const float S32 = __uint_as_float((uint32_t)(key >> 32));
    if (history != nullptr) history[pc.iters] = S32;
    for (int d = 0; d < AFM_MAXD; ++d)
        w->x[d] = d < pc.D ? (double)sw.pb[fin][(size_t)d * pc.P + g] : 0.0;
    w->S32 = S32;
    w->winner = g;
}

// The lowest of Kn misfits (first index on ties); x [D][Kn]; idx maps the
// candidate to its swarm index (or nullptr).  One thread.
__global__ void reeval_pick_min_kernel(int D, int Kn, const float* __restrict__ x,
                                       const float* __restrict__ S, const int* __restrict__ idx,
                                       ReevalWinner* __restrict__ w) {
    int kb = 0;
    for (int k = 1; k < Kn; ++k)
        if (S[k] < S[kb]) kb = k;
    for (int d = 0; d < AFM_MAXD; ++d) w->x[d] = d < D ? (double)x[(size_t)d * Kn + kb] : 0.0;
    w->S32 = S[kb];
    w->winner = idx != nullptr ? idx[kb] : kb;
}

// Drive tables, sum of U^2, FP64 force coefficients of the winner, and the
// FP32 guess of the segment start states (start[0]; b = 0 is the exact FP64
// initial state).
template <int M, int FORCE>
__global__ void __launch_bounds__(256) reeval_guess_kernel(const KAffine<float> Kf,
                                                           const KAffine<double> Kd,
                                                           const ReevalPtrs R,
                                                           const float* __restrict__ U) {
    extern __shared__ __align__(16) float tabf[];
    __shared__ double red[256];
    aff::build_rows<float, M, FORCE>(Kf, tabf);
    const int spc = Kd.spc2 >> 1;
    for (int j = threadIdx.x; j < spc; j += blockDim.x)
        sincospi((2.0 / (double)spc) * (double)j, &R.tab[2 * j], &R.tab[2 * j + 1]);
    double acc = 0.0;
    const int nv = Kd.n_steps * (Kd.np > 0 ? Kd.np : 1);   // record values
    for (int n = threadIdx.x; n < nv; n += blockDim.x) acc += (double)U[n] * (double)U[n];
    red[threadIdx.x] = acc;
    __syncthreads();
    for (int s = blockDim.x / 2; s > 0; s >>= 1) {
        if ((int)threadIdx.x < s) red[threadIdx.x] += red[threadIdx.x + s];
        __syncthreads();
    }
    constexpr int S2 = 2 * M;
    double* Y = R.start[0];
    if (threadIdx.x == 0) {
        *R.sumU2 = red[0];
        ReevalWinner* w = R.win;
        double xd[AFM_MAXD];
        for (int d = 0; d < AFM_MAXD; ++d) xd[d] = w->x[d];
        const Coef<double> cd = make_coef<double, double>(Kd, xd);
        w->c[0] = cd.c0;
        w->c[1] = cd.c1;
        w->c[2] = cd.c2;
        w->c[3] = cd.c3;
        const Coef<float> c = make_coef<float, double>(Kf, xd);
#pragma unroll
        for (int i = 0; i < M; ++i) {
            Y[i] = Kd.q0[i];
            Y[M + i] = Kd.v0[i];
        }
        guess_starts<M, FORCE>(Kf, c, tabf, R.B, Y);
    }
    __syncthreads();
    for (int b = 1 + threadIdx.x; b < R.B; b += blockDim.x)
        finish_start<M>(Kd, Y + (size_t)b * S2);
}

// One thread per segment b: AFM_SEG FP64 steps from Z_b -> E_b and the
// segment's misfit share Sb_b; TANGENT: also J_b ([2m][2m], row = output
// component, column = input direction) in FP32 from the recorded slopes.
template <int M, int FORCE, bool TANGENT>
__global__ void __launch_bounds__(32) reeval_pass_kernel(const KAffine<double> K,
                                                         const ReevalPtrs R,
                                                         const double* __restrict__ Z,
                                                         const float* __restrict__ U) {
    __shared__ float rec[TANGENT ? AFM_SEG * kRec * 32 : 1];
    constexpr int S2 = 2 * M;
    const int lane = threadIdx.x;
    const int b = blockIdx.x * 32 + lane;
    if (b >= R.B) return;
    const Coef<double> cw = winner_coef(*R.win);
    const aff::LawCoef<double> c = aff::law_coef(cw);
    Coef<float> cf;
    cf.c0 = (float)cw.c0;
    cf.c1 = (float)cw.c1;
    cf.c2 = (float)cw.c2;
    cf.c3 = (float)cw.c3;
    aff::State<double, M, aff::NONE> st;
    aff::import_state<M>(K, Z + (size_t)b * S2, Z + (size_t)b * S2 + M, st);
    const int n0 = b * AFM_SEG;
    const int n1 = min(n0 + AFM_SEG, K.n_steps);
    const int spc = K.spc2 >> 1;
    int j = n0 % spc;
    double S = 0.0;
    for (int s = n0; s < n1; ++s) {
        double r[aff::Rows<M, FORCE>::words];
        drive_terms<M, FORCE, true>(K, R.tab, j, r);
        if (++j == spc) j = 0;
        step64<M, FORCE, TANGENT>(K, c, cf, r, st, rec + lane + (s - n0) * kRec * 32);
        if (K.np > 0) {   // deflection points
            for (int k = 0; k < K.np; ++k) {
                const double e = (double)U[(size_t)s * K.np + k] - aff::point_defl(K, k, st);
                S = fma(e, e, S);
            }
        } else {
            const double e = (double)U[s] - aff::tip(st);
            S = fma(e, e, S);
        }
    }
    double q[M], v[M];
    aff::export_state<double, M, aff::NONE>(K, st, q, v);
#pragma unroll
    for (int i = 0; i < M; ++i) {
        R.E[(size_t)b * S2 + i] = q[i];
        R.E[(size_t)b * S2 + M + i] = v[i];
    }
    R.Sb[b] = S;
    if (TANGENT) {
        float w2[M], wq[M], tip[M];
#pragma unroll
        for (int i = 0; i < M; ++i) {
            w2[i] = (float)K.w2[i];
            wq[i] = (float)K.wq[i];
            tip[i] = (float)K.tip[i];
        }
        const int ns = n1 - n0;
#pragma unroll 1
        for (int col = 0; col < S2; ++col) {
            float dq[M], dv[M];
#pragma unroll
            for (int i = 0; i < M; ++i) {
                dq[i] = col == i ? 1.f : 0.f;
                dv[i] = col == M + i ? 1.f : 0.f;
            }
            for (int t = 0; t < ns; ++t) jvp_step<M, FORCE>(w2, wq, tip, rec + lane + t * kRec * 32, dq, dv);
            double* Jc = R.J + (size_t)b * S2 * S2 + col;
#pragma unroll
            for (int i = 0; i < M; ++i) {
                Jc[i * S2] = (double)dq[i];
                Jc[(M + i) * S2] = (double)dv[i];
            }
        }
    }
}

template <int M>
__global__ void __launch_bounds__(32) reeval_correct_kernel(const ReevalPtrs R,
                                                            const double* __restrict__ Zold,
                                                            double* __restrict__ Znew) {
    correct_starts<M>(Zold, Znew, R.E, R.J, R.B);
}

// S_f64 = sum of the segment shares, the join check (with the sequential
// fallback) and the result record.  One block of 256.
template <int M, int FORCE>
__global__ void __launch_bounds__(256) reeval_final_kernel(const KAffine<double> K,
                                                           const ReevalPtrs R,
                                                           const double* __restrict__ Z,
                                                           const float* __restrict__ U, int iters,
                                                           const int* __restrict__ flags,
                                                           afm_result* __restrict__ res) {
    __shared__ double rs[256], rd[256];
    constexpr int S2 = 2 * M;
    double s = 0.0, dsum = 0.0;
    for (int b = threadIdx.x; b < R.B; b += blockDim.x) {
        s += R.Sb[b];
        if (b + 1 < R.B) {
            double mx = 0.0;
#pragma unroll
            for (int i = 0; i < S2; ++i) {
                const double e = fabs(R.E[(size_t)b * S2 + i] - Z[(size_t)(b + 1) * S2 + i]);
                if (!(e <= mx)) mx = e;   // keeps a NaN
            }
            dsum += mx;
        }
    }
    rs[threadIdx.x] = s;
    rd[threadIdx.x] = dsum;
    __syncthreads();
    for (int h = blockDim.x / 2; h > 0; h >>= 1) {
        if ((int)threadIdx.x < h) {
            rs[threadIdx.x] += rs[threadIdx.x + h];
            rd[threadIdx.x] += rd[threadIdx.x + h];
        }
        __syncthreads();
    }
    if (threadIdx.x != 0) return;
    const ReevalWinner& w = *R.win;
    double S64 = rs[0];
    const double defect = rd[0];
    int segs = R.B;
    if (!(defect <= kDefectTol) || !isfinite(S64)) {
        S64 = integrate64<M, FORCE, true>(K, aff::law_coef(winner_coef(w)), R.tab, U, K.n_steps);
        segs = 0;
    }
    double th[AFM_MAXD];
    for (int s5 = 0; s5 < AFM_MAXD; ++s5) th[s5] = K.fixed[s5];
    for (int d = 0; d < K.D; ++d) {
        const double v = K.lo[d] + w.x[d] * K.span[d];
        th[K.slot[d]] = K.logs[d] ? exp10(v) : v;
    }
    for (int d = 0; d < AFM_MAXD; ++d) {
        res->x[d] = w.x[d];
        res->theta[d] = th[d];
    }
    const double u2 = *R.sumU2;
    res->S = (double)w.S32;
    res->S_f64 = S64;
    res->J_rel = u2 > 0.0 ? sqrt(S64 / u2) : 0.0;
    res->iters = iters;
    res->winner = w.winner;
    res->nonfinite = flags != nullptr ? flags[0] : 0;
    res->status = (isfinite(S64) && res->nonfinite == 0) ? AFM_OK : AFM_ERR_NONFINITE;
    res->defect = segs > 0 ? defect : (defect <= kDefectTol ? 0.0 : defect);
    res->segments = segs;
    res->reserved = 0;
    for (int k = 0; k < 3; ++k) res->drive[k] = 0.0;
}

// ---------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------
bool reeval_supported(int m, int n_steps) {
    return m >= 1 && m <= AFM_MAXM && n_steps >= 2 * AFM_SEG;
}


size_t reeval_bytes(int m, int n_steps, int spc) {
    const size_t B = (size_t)reeval_segments(n_steps), S2 = 2 * (size_t)reeval_modes(m);
    return a256(sizeof(ReevalWinner)) + a256(sizeof(double) * (2 * (size_t)spc + 1)) +
           2 * a256(sizeof(double) * (B + 1) * S2) + a256(sizeof(double) * B * S2) +
           a256(sizeof(double) * B * S2 * S2) + a256(sizeof(double) * B) + 256;
}

void reeval_carve(void* base, int m, int n_steps, int spc, ReevalPtrs* R) {
    const size_t B = (size_t)reeval_segments(n_steps), S2 = 2 * (size_t)reeval_modes(m);
    char* p = static_cast<char*>(base);
    R->win = reinterpret_cast<ReevalWinner*>(p);
    p += a256(sizeof(ReevalWinner));
    R->tab = reinterpret_cast<double*>(p);
    p += a256(sizeof(double) * (2 * (size_t)spc + 1));
    R->start[0] = reinterpret_cast<double*>(p);
    p += a256(sizeof(double) * (B + 1) * S2);
    R->start[1] = reinterpret_cast<double*>(p);
    p += a256(sizeof(double) * (B + 1) * S2);
    R->E = reinterpret_cast<double*>(p);
    p += a256(sizeof(double) * B * S2);
    R->J = reinterpret_cast<double*>(p);
    p += a256(sizeof(double) * B * S2 * S2);
    R->Sb = reinterpret_cast<double*>(p);
    p += a256(sizeof(double) * B);
    R->sumU2 = reinterpret_cast<double*>(p);
    R->B = (int)B;
}

cudaError_t launch_reeval_pick_swarm(const PsoConst& pc, const SwarmPtrs& sw, float* history,
                                     ReevalWinner* w, cudaStream_t st) {
    reeval_pick_swarm_kernel<<<1, 1, 0, st>>>(pc, sw, history, w);
    return cudaGetLastError();
}

cudaError_t launch_reeval_pick_min(int D, int Kn, const float* x, const float* S, const int* idx,
                                   ReevalWinner* w, cudaStream_t st) {
    reeval_pick_min_kernel<<<1, 1, 0, st>>>(D, Kn, x, S, idx, w);
    return cudaGetLastError();
}

cudaError_t launch_reeval(const KAffine<float>& Kf, const KAffine<double>& Kd, const ReevalPtrs& R,
                          const float* U, int iters, const int* flags, void* result,
                          cudaStream_t st) {
    if (!reeval_supported(Kd.m, Kd.n_steps) || R.B != reeval_segments(Kd.n_steps))
        return cudaErrorInvalidValue;
    return dispatch_m13(Kd.m, Kd.force, [&](auto Mc, auto Fc) -> cudaError_t {
        constexpr int M = decltype(Mc)::value, FORCE = decltype(Fc)::value;
        const size_t smem = aff_table_bytes<float, M, FORCE>(Kf.spc2);
        cudaError_t e = cudaSuccess;
        if (smem > 40 * 1024)
            e = cudaFuncSetAttribute(reeval_guess_kernel<M, FORCE>,
                                     cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        reeval_guess_kernel<M, FORCE><<<1, 256, smem, st>>>(Kf, Kd, R, U);
        e = cudaGetLastError();
        const int grid = (R.B + 31) / 32;
        for (int k = 0; e == cudaSuccess && k < kSweeps; ++k) {
            reeval_pass_kernel<M, FORCE, true><<<grid, 32, 0, st>>>(Kd, R, R.start[k & 1], U);
            if ((e = cudaGetLastError()) != cudaSuccess) break;
            reeval_correct_kernel<M><<<1, 32, 0, st>>>(R, R.start[k & 1], R.start[(k + 1) & 1]);
            e = cudaGetLastError();
        }
        if (e != cudaSuccess) return e;
        const double* Zf = R.start[kSweeps & 1];
        reeval_pass_kernel<M, FORCE, false><<<grid, 32, 0, st>>>(Kd, R, Zf, U);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        reeval_final_kernel<M, FORCE><<<1, 256, 0, st>>>(Kd, R, Zf, U, iters, flags,
                                                         reinterpret_cast<afm_result*>(result));
        return cudaGetLastError();
    });
}

}  // namespace afm
