// kern_lm.cu -- Levenberg-Marquardt polish: residual sensitivities by
// tangent-linear (forward-mode) differentiation of the FP32 RK4 solve, the
// normal equations of the misfit (Eq. 5), damped Gauss-Newton trial points
// for a ladder of damping values, and the choice among them.
//
// For the misfit S = sum_n r_n^2, r_n = U_n - u_n(x), the sensitivities
// a_n = du_n/dx (D per step) give H = sum a_n a_n^T (Gauss-Newton matrix,
// half the Gauss-Newton Hessian) and b = sum a_n r_n = -dS/dx / 2.  The
// primal solve inside the sensitivity kernel is the forward kernel's
// arithmetic, so S is bit-identical to afm_forward_batch's.
#include <type_traits>

#include "afm_device.cuh"
#include "afm_launch.h"
#include "afm_tangent.cuh"
#include "afm_warp.cuh"
#include "kern_lm.cuh"

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

constexpr int kThreads = 128;   // (32: the drive table, built by one warp, costs 10 % more)
constexpr int kFold = 32;   // steps summed in FP32 before folding into FP64 totals

}  // namespace

// Sensitivity pass of one particle per thread: S (as the forward kernel),
// H [P][D][D] and b [P][D] in FP64.  CS: the tangents run along the law's
// coefficients (afm_tangent.cuh), else along ND free parameters.  Ragged
// form as the adjoint: off != nullptr gives particle p the record of pixel
// order[p / per_slot].
// PP (ragged form only): each particle's pixel has its own constants and
// drive table (pix), read from global memory.
// FMA-pipe bound when wide: DMT with 3 modes issues ~380 FP32 operations per
// step (147 the solve, ~30 the partials, 3 x 65 the tangents, 9 the sums;
// ~640 with parameter directions and linearised stages).  16 384 candidates x
// 1 280 steps: 432 us, 696 us so.
template <int M, int FORCE, int ND, bool CS, bool PP>
__global__ void __launch_bounds__(kThreads) sens_kernel(const KAffine<float> K0,
                                                        const float* __restrict__ x, int P,
                                                        const float* __restrict__ U,
                                                        const int64_t* __restrict__ off,
                                                        const int* __restrict__ order,
                                                        int per_slot, float* __restrict__ S_out,
                                                        double* __restrict__ H_out,
                                                        double* __restrict__ b_out,
                                                        const PixConst pixc) {
    constexpr int NH = ND * (ND + 1) / 2, NC = aff::CoefDirs<FORCE>::n;
    static_assert(!CS || ND == NC, "coefficient directions");
    extern __shared__ __align__(16) float tabs[];
    __shared__ double accH[NH][kThreads], accb[ND][kThreads];
    if constexpr (!PP) {
        build_drive_table(K0, tabs);
        __syncthreads();
    }
    const int tid = threadIdx.x;
    const int p = blockIdx.x * blockDim.x + tid;
    if (p >= P) return;
    int n = K0.n_steps, pix = 0;
    if (off != nullptr) {
        const int slot = p / per_slot;
        pix = order != nullptr ? order[slot] : slot;
        U += off[pix];
        n = (int)(off[pix + 1] - off[pix]);
    }
    const KAffine<float>* Kp = &K0;
    const float* tab = tabs;
    if constexpr (PP) {
        Kp = pixc.kf + pix;
        tab = pixc.tab32 + (size_t)pix * pixc.ld;
    }
    const KAffine<float>& K = *Kp;
    const int D = K.D;
    float xd[AFM_MAXD];
    for (int d = 0; d < AFM_MAXD; ++d) xd[d] = d < D ? x[(size_t)d * P + p] : 0.f;
    const Coef<float> c = make_coef<float, float>(K, xd);
    float Jc[NC][CS ? 1 : ND];
    if constexpr (!CS) {
        double Jd[4][AFM_MAXD];
        coef_jacobian<float>(K, xd, Jd);
#pragma unroll
        for (int k = 0; k < NC; ++k)
#pragma unroll
            for (int e = 0; e < ND; ++e)
                Jc[k][e] = e < D ? (float)Jd[aff::CoefDirs<FORCE>::index(k)][e] : 0.f;
    }
    const warp::Modes<M> C = warp::modes<M>(K);
    warp::State<M> st;
    warp::init<M>(K, C, tab[0], st);
    aff::Tangent<M> tg[ND];
#pragma unroll
    for (int e = 0; e < ND; ++e) aff::zero(tg[e]);
#pragma unroll
    for (int t = 0; t < NH; ++t) accH[t][tid] = 0.0;
#pragma unroll
    for (int e = 0; e < ND; ++e) accb[e][tid] = 0.0;
    float hc[NH], bc[ND];
#pragma unroll
    for (int t = 0; t < NH; ++t) hc[t] = 0.f;
#pragma unroll
    for (int e = 0; e < ND; ++e) bc[e] = 0.f;
    float S = 0.f, cS = 0.f;
    int j = 0, fold = 0;
    const int spc2 = K.spc2;
    float Un = n > 0 ? U[0] : 0.f;
    for (int s = 0; s < n; ++s) {
        const float gh = tab[j + 1], g1 = tab[j + 2];
        j += 2;
        if (j >= spc2) j = 0;
        const float Unext = s + 1 < n ? U[s + 1] : 0.f;
        warp::Gaps g;
        warp::step<M, FORCE>(C, c, gh, g1, st, g);
        aff::Partials<FORCE> Ps[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) aff::partials<FORCE>(c, g.d[k], g.r[k], Ps[k]);
        const float r = __fsub_rn(Un, st.u);
        warp::misfit_add(Un, st.u, S, cS);
        Un = Unext;
#pragma unroll
        for (int e = 0; e < ND; ++e) {
            float G[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                if constexpr (CS) {
                    G[k] = Ps[k].Fc[e];
                } else {
                    G[k] = aff::mul(Ps[k].Fc[0], Jc[0][e]);
#pragma unroll
                    for (int l = 1; l < NC; ++l) G[k] = aff::fma(Ps[k].Fc[l], Jc[l][e], G[k]);
                }
            }
            aff::tangent_step<M, FORCE>(K, Ps, G, tg[e]);
        }
        int w = 0;
#pragma unroll
        for (int e = 0; e < ND; ++e) {
            const float ae = aff::tip(tg[e]);
            bc[e] = aff::fma(ae, r, bc[e]);
#pragma unroll
            for (int f = 0; f <= e; ++f) {
                hc[w] = aff::fma(ae, aff::tip(tg[f]), hc[w]);
                ++w;
            }
        }
        if (++fold == kFold || s + 1 == n) {
            fold = 0;
#pragma unroll
            for (int t2 = 0; t2 < NH; ++t2) {
                accH[t2][tid] += (double)hc[t2];
                hc[t2] = 0.f;
            }
#pragma unroll
            for (int e = 0; e < ND; ++e) {
                accb[e][tid] += (double)bc[e];
                bc[e] = 0.f;
            }
        }
    }
    if (!(S < INFINITY)) S = INFINITY;
    S_out[p] = S;
    double* H = H_out + (size_t)p * D * D;
    double* b = b_out + (size_t)p * D;
    if constexpr (CS) {
        double Hc[NH], bd[ND], Jd[4][AFM_MAXD];
        coef_jacobian<float>(K, xd, Jd);
#pragma unroll
        for (int t = 0; t < NH; ++t) Hc[t] = accH[t][tid];
#pragma unroll
        for (int e = 0; e < ND; ++e) bd[e] = accb[e][tid];
        for (int e = 0; e < D; ++e) aff::map_row<FORCE>(Jd, Hc, bd, D, e, H, b);
    } else {
        int w = 0;
        for (int e = 0; e < ND; ++e) {
            for (int f = 0; f <= e; ++f) {
                if (e < D) {
                    H[e * D + f] = accH[w][tid];
                    H[f * D + e] = accH[w][tid];
                }
                ++w;
            }
            if (e < D) b[e] = accb[e][tid];
        }
    }
}

// Trial points of candidate k: clamp(x + delta_j) with (H + lambda_j W)
// delta_j = b, lambda_j = lam0 ratio^j, W = diag(max(H_dd, 1e-12 max H_ee)),
// solved by Cholesky in FP64.  Output column k * J + j of Xc [D][K*J].
__global__ void lm_cand_kernel(int D, int K, int J, const float* __restrict__ x,
                               const double* __restrict__ H, const double* __restrict__ b,
                               double lam0, double ratio, float* __restrict__ Xc) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= K) return;
    const double* Hk = H + (size_t)k * D * D;
    double hmax = 0.0;
    for (int d = 0; d < D; ++d) hmax = fmax(hmax, Hk[d * D + d]);
    const size_t KJ = (size_t)K * J;
    double lam = lam0;
    for (int j = 0; j < J; ++j, lam *= ratio) {
        double L[AFM_MAXD][AFM_MAXD], y[AFM_MAXD];
        bool ok = hmax > 0.0;
        for (int r = 0; r < D && ok; ++r) {
            for (int c = 0; c <= r; ++c) {
                double s = Hk[r * D + c];
                if (r == c) s += lam * fmax(Hk[r * D + r], 1e-12 * hmax);
                for (int t = 0; t < c; ++t) s -= L[r][t] * L[c][t];
                if (r == c) {
                    if (!(s > 0.0)) {
                        ok = false;
                        break;
                    }
                    L[r][r] = sqrt(s);
                } else {
                    L[r][c] = s / L[c][c];
                }
            }
        }
        if (ok) {
            for (int r = 0; r < D; ++r) {
                double s = b[(size_t)k * D + r];
                for (int t = 0; t < r; ++t) s -= L[r][t] * y[t];
                y[r] = s / L[r][r];
            }
            for (int r = D - 1; r >= 0; --r) {
                double s = y[r];
                for (int t = r + 1; t < D; ++t) s -= L[t][r] * y[t];
                y[r] = s / L[r][r];
            }
        }
        for (int d = 0; d < D; ++d) {
            double xn = (double)x[(size_t)d * K + k] + (ok ? y[d] : 0.0);
            if (!(xn > 0.0)) xn = 0.0;
            if (xn > 1.0) xn = 1.0;
            Xc[(size_t)d * KJ + (size_t)k * J + j] = (float)xn;
        }
    }
}

// The trial point of least misfit (first on ties) replaces x if it lowers S.
__global__ void lm_select_kernel(int D, int K, int J, float* __restrict__ x, float* __restrict__ S,
                                 const float* __restrict__ Xc, const float* __restrict__ Sc) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= K) return;
    int jb = 0;
    for (int j = 1; j < J; ++j)
        if (Sc[(size_t)k * J + j] < Sc[(size_t)k * J + jb]) jb = j;
    const float Sj = Sc[(size_t)k * J + jb];
    if (Sj < S[k]) {
        const size_t KJ = (size_t)K * J;
        for (int d = 0; d < D; ++d) x[(size_t)d * K + k] = Xc[(size_t)d * KJ + (size_t)k * J + jb];
        S[k] = Sj;
    }
}

// lm_select_kernel for the fused step: the point kept also brings its normal
// equations (computed by the sensitivity pass over the trial points).
__global__ void lm_select_hb_kernel(int D, int K, int J, float* __restrict__ x, float* __restrict__ S,
                                    double* __restrict__ H, double* __restrict__ b,
                                    const float* __restrict__ Xc, const float* __restrict__ Sc,
                                    const double* __restrict__ Hc, const double* __restrict__ bc) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= K) return;
    int jb = 0;
    for (int j = 1; j < J; ++j)
        if (Sc[(size_t)k * J + j] < Sc[(size_t)k * J + jb]) jb = j;
    const float Sj = Sc[(size_t)k * J + jb];
    if (Sj < S[k]) {
        const size_t KJ = (size_t)K * J, c = (size_t)k * J + jb;
        for (int d = 0; d < D; ++d) x[(size_t)d * K + k] = Xc[(size_t)d * KJ + c];
        for (int e = 0; e < D * D; ++e) H[(size_t)k * D * D + e] = Hc[c * D * D + e];
        for (int d = 0; d < D; ++d) b[(size_t)k * D + d] = bc[c * D + d];
        S[k] = Sj;
    }
}

cudaError_t launch_lm_select_hb(int D, int K, int J, float* x, float* S, double* H, double* b,
                                const float* Xc, const float* Sc, const double* Hc,
                                const double* bc, cudaStream_t st) {
    const int threads = 64;
    lm_select_hb_kernel<<<(K + threads - 1) / threads, threads, 0, st>>>(D, K, J, x, S, H, b, Xc,
                                                                         Sc, Hc, bc);
    return cudaGetLastError();
}

cudaError_t launch_sens(const KAffine<float>& K, const float* x, int P, const float* U, float* S,
                        double* H, double* b, cudaStream_t st, const int64_t* off, const int* order,
                        int per_slot, const PixConst& pix) {
    const bool pp = pix.kf != nullptr;
    if (pp && off == nullptr) return cudaErrorInvalidValue;
    if (!pp && sens_lanes_preferred(P, K.D))
        return launch_sens_lanes(K, x, P, U, S, H, b, st, off, order, per_slot);
    const int blocks = (P + kThreads - 1) / kThreads;
    return dispatch_mf(K.m, K.force, [&](auto Mc, auto Fc) -> cudaError_t {
        constexpr int M = decltype(Mc)::value, FORCE = decltype(Fc)::value;
        const size_t smem = pp ? 0 : sizeof(float) * (size_t)(K.spc2 + 1);
        auto go = [&](auto Dc, auto Cc, auto Pc) -> cudaError_t {
            auto kern = sens_kernel<M, FORCE, decltype(Dc)::value, decltype(Cc)::value,
                                    decltype(Pc)::value>;
            if (smem > 24 * 1024) {
                cudaError_t e = cudaFuncSetAttribute(
                    kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
                if (e != cudaSuccess) return e;
            }
            kern<<<blocks, kThreads, smem, st>>>(K, x, P, U, off, order, per_slot, S, H, b, pix);
            return cudaGetLastError();
        };
        return sens_dirs<FORCE>(K.D, [&](auto Dc, auto Cc) -> cudaError_t {
            return pp ? go(Dc, Cc, std::true_type{}) : go(Dc, Cc, std::false_type{});
        });
    });
}

cudaError_t launch_lm_cand(int D, int K, int J, const float* x, const double* H, const double* b,
                           double lam0, double ratio, float* Xc, cudaStream_t st) {
    const int threads = 64;
    lm_cand_kernel<<<(K + threads - 1) / threads, threads, 0, st>>>(D, K, J, x, H, b, lam0, ratio, Xc);
    return cudaGetLastError();
}

cudaError_t launch_lm_select(int D, int K, int J, float* x, float* S, const float* Xc,
                             const float* Sc, cudaStream_t st) {
    const int threads = 64;
    lm_select_kernel<<<(K + threads - 1) / threads, threads, 0, st>>>(D, K, J, x, S, Xc, Sc);
    return cudaGetLastError();
}

}  // namespace afm
