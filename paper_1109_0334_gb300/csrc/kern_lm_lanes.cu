// kern_lm_lanes.cu -- the sensitivity pass of kern_lm.cu with the tangent
// directions of a candidate spread over L lanes (one direction per lane),
// for candidate counts too small to fill the GPU (the polish of one
// inversion's best particles).  Every lane runs the primal solve
// (identical arithmetic, so S is the forward kernel's bit for bit) and the
// tangent of its own direction; each step the group gathers the tip
// tangents with shuffles and lane e accumulates row e of H = sum a a^T and
// b_e = sum a_e r.  Each direction's arithmetic, every accumulation and the
// final map to the parameters are the one-lane kernel's operations in the
// same order, so H and b are bit-identical to sens_kernel's.
//
// Bound by one warp's instruction stream (~300 per step for DMT, 3 modes):
// the tangent of a step runs beside the primal of the next, which fills the
// gaps of both chains.  512 candidates x 2 560 steps: 589 us (834 us with
// primal and tangent of one step in turn, 895 us with one lane per
// (direction, mode) pair and twelve groups of shuffles per step).
#include <type_traits>

#include "afm_device.cuh"
#include "afm_launch.h"
#include "afm_tangent.cuh"
#include "afm_warp.cuh"
#include "kern_lm.cuh"

namespace afm {

namespace {

// Threads of a block: the first wpb warps carry candidates, all of them build
// the drive table.
constexpr int kLaneThreads = 128;
constexpr int kLaneFold = 32;   // as sens_kernel: FP32 blocks of 32 steps folded into FP64

}  // namespace

// RAG: ragged form (off != nullptr), the lanes of a warp follow records of
// different lengths; else one record for all.
template <int M, int FORCE, int ND, bool CS, bool RAG>
__global__ void __launch_bounds__(kLaneThreads) sens_lanes_kernel(
    const KAffine<float> K, const float* __restrict__ x, int P, const float* __restrict__ U,
    const int64_t* __restrict__ off, const int* __restrict__ order, int per_slot, int wpb,
    float* __restrict__ S_out, double* __restrict__ H_out, double* __restrict__ b_out) {
    constexpr int L = ND <= 2 ? 2 : 4, NC = aff::CoefDirs<FORCE>::n;
    constexpr int NH = ND * (ND + 1) / 2, G = kLaneThreads / L;
    extern __shared__ __align__(16) float tab[];
    __shared__ double sH[G][NH], sb[G][ND];
    build_drive_table(K, tab);
    __syncthreads();
    const int lane = threadIdx.x & 31;
    if ((int)threadIdx.x >= 32 * wpb) return;   // whole warps
    const int p0 = blockIdx.x * (wpb * 32 / L) + threadIdx.x / L, grp = threadIdx.x / L;
    if (p0 - lane / L >= P) return;
    const int ln = lane % L, e = ln < ND ? ln : 0;   // this lane's direction (a spare lane repeats 0)
    const bool store = p0 < P;
    const int p = min(p0, P - 1);            // groups past P repeat the last candidate
    const int D = K.D;
    int n = K.n_steps;
    if constexpr (RAG) {
        const int slot = p / per_slot;
        const int pix = order != nullptr ? order[slot] : slot;
        U += off[pix];
        n = (int)(off[pix + 1] - off[pix]);
    }
    // the whole warp steps to its longest record (groups with shorter records
    // run on without summing), so that every shuffle has the full warp
    int n_warp = n;
    if constexpr (RAG) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
            n_warp = max(n_warp, __shfl_xor_sync(0xffffffffu, n_warp, o));
    }
    float xd[AFM_MAXD];
    for (int d = 0; d < AFM_MAXD; ++d) xd[d] = d < D ? x[(size_t)d * P + p] : 0.f;
    const Coef<float> c = make_coef<float, float>(K, xd);
    float Jc[NC];
    if constexpr (!CS) {
        double Jd[4][AFM_MAXD];
        coef_jacobian<float>(K, xd, Jd);
#pragma unroll
        for (int k = 0; k < NC; ++k) {
            float jk = 0.f;
            for (int d = 0; d < AFM_MAXD; ++d)
                if (d == e && d < D) jk = (float)Jd[aff::CoefDirs<FORCE>::index(k)][d];
            Jc[k] = jk;
        }
    }
    const warp::Modes<M> C = warp::modes<M>(K);
    warp::State<M> st;
    warp::init<M>(K, C, tab[0], st);
    aff::Tangent<M> tg;
    aff::zero(tg);
    double aH[ND], ab = 0.0;
#pragma unroll
    for (int f = 0; f < ND; ++f) aH[f] = 0.0;
    float S = 0.f, cS = 0.f;
    const int spc2 = K.spc2;
    int j = 0;
    float gh = tab[1], g1 = tab[2];
    // the partials of the step whose tangent comes next: the force slopes, and
    // the force terms of this lane's direction
    aff::Partials<FORCE> Ps[4];
    float Gs[4], r = 0.f;
    auto primal = [&](float Un, bool sum) {
        warp::Gaps g;
        warp::step<M, FORCE>(C, c, gh, g1, st, g);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            aff::partials<FORCE>(c, g.d[k], g.r[k], Ps[k]);
            if constexpr (CS) {
                Gs[k] = Ps[k].Fc[0];
#pragma unroll
                for (int l = 1; l < NC; ++l) Gs[k] = e == l ? Ps[k].Fc[l] : Gs[k];
            } else {
                Gs[k] = aff::mul(Ps[k].Fc[0], Jc[0]);
#pragma unroll
                for (int l = 1; l < NC; ++l) Gs[k] = aff::fma(Ps[k].Fc[l], Jc[l], Gs[k]);
            }
        }
        r = __fsub_rn(Un, st.u);
        if (sum) warp::misfit_add(Un, st.u, S, cS);
    };
    // record values: one record is read 32 values at a time, a block ahead, one
    // per lane; ragged records one step ahead
    float Ub = (!RAG && lane < n) ? U[lane] : 0.f;
    float Un = n > 0 ? U[0] : 0.f;
    primal(Un, n > 0);
    if (RAG) Un = n > 1 ? U[1] : 0.f;
    // tangent of step s beside the primal step s + 1 (they are independent, so
    // their chains fill each other's gaps), in blocks of kLaneFold steps summed
    // in FP32 and folded into the FP64 totals
    for (int s0 = 0; s0 < n_warp; s0 += kLaneFold) {
        const int kn = s0 + kLaneFold + lane;
        const float Unb = (!RAG && kn < n) ? U[kn] : 0.f;
        const int cnt = min(kLaneFold, n_warp - s0);
        float hc[ND], bc = 0.f;
#pragma unroll
        for (int f = 0; f < ND; ++f) hc[f] = 0.f;
        for (int k = 0; k < cnt; ++k) {
            const int s = s0 + k;
            j += 2;
            if (j >= spc2) j = 0;
            gh = tab[j + 1];
            g1 = tab[j + 2];
            // the record value of step s + 1
            float Us = Un;
            if constexpr (RAG)
                Un = s + 2 < n ? U[s + 2] : 0.f;
            else
                Us = __shfl_sync(0xffffffffu, k + 1 < kLaneFold ? Ub : Unb, (k + 1) & 31);
            const float rs = r;
            aff::tangent_step<M, FORCE>(K, Ps, Gs, tg);
            const float au = aff::tip(tg);
            float af[ND];
#pragma unroll
            for (int f = 0; f < ND; ++f) af[f] = __shfl_sync(0xffffffffu, au, f, L);
            primal(Us, s + 1 < n);
            if (!RAG || s < n) {
                bc = aff::fma(au, rs, bc);
#pragma unroll
                for (int f = 0; f < ND; ++f) hc[f] = aff::fma(au, af[f], hc[f]);
            }
        }
#pragma unroll
        for (int f = 0; f < ND; ++f) aH[f] += (double)hc[f];
        ab += (double)bc;
        Ub = Unb;
    }
    if (ln < ND) {
#pragma unroll
        for (int f = 0; f < ND; ++f)
            if (f <= e) sH[grp][e * (e + 1) / 2 + f] = aH[f];
        sb[grp][e] = ab;
    }
    __syncwarp();
    if (!store) return;
    if (ln == 0) S_out[p] = (S < INFINITY) ? S : INFINITY;
    double* H = H_out + (size_t)p * D * D;
    double* b = b_out + (size_t)p * D;
    if constexpr (CS) {
        double Jd[4][AFM_MAXD];
        coef_jacobian<float>(K, xd, Jd);
        for (int row_e = ln; row_e < D; row_e += L)
            aff::map_row<FORCE>(Jd, sH[grp], sb[grp], D, row_e, H, b);
    } else if (ln < ND && e < D) {
        for (int f = 0; f <= e; ++f) {
            H[e * D + f] = sH[grp][e * (e + 1) / 2 + f];
            H[f * D + e] = sH[grp][e * (e + 1) / 2 + f];
        }
        b[e] = sb[grp][e];
    }
}

// One warp per SM sub-partition at most: past that the redundant primal
// solves cost more than the shorter chains gain.
bool sens_lanes_preferred(int P, int D) {
    const int L = D <= 2 ? 2 : 4;
    return (long long)P * L <= 152LL * 4 * 32;
}

cudaError_t launch_sens_lanes(const KAffine<float>& K, const float* x, int P, const float* U,
                              float* S, double* H, double* b, cudaStream_t st, const int64_t* off,
                              const int* order, int per_slot) {
    auto byM = [&](auto Mc, auto Fc) -> cudaError_t {
        constexpr int M = decltype(Mc)::value, FORCE = decltype(Fc)::value;
        const size_t smem = sizeof(float) * (size_t)(K.spc2 + 1);
        return sens_dirs<FORCE>(K.D, [&](auto Dc, auto Cc) -> cudaError_t {
            constexpr int ND = decltype(Dc)::value, L = ND <= 2 ? 2 : 4;
            constexpr bool CS = decltype(Cc)::value;
            auto kern = off != nullptr ? sens_lanes_kernel<M, FORCE, ND, CS, true>
                                       : sens_lanes_kernel<M, FORCE, ND, CS, false>;
            if (smem > 24 * 1024) {
                cudaError_t e = cudaFuncSetAttribute(
                    kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
                if (e != cudaSuccess) return e;
            }
            const int warps = (int)(((long long)P * L + 31) / 32);
            const int wpb = warps <= 152 ? 1 : warps <= 304 ? 2 : 4;
            kern<<<(warps + wpb - 1) / wpb, kLaneThreads, smem, st>>>(K, x, P, U, off, order,
                                                                       per_slot, wpb, S, H, b);
            return cudaGetLastError();
        });
    };
    auto byF = [&](auto Mc) -> cudaError_t {
        switch (K.force) {
            case F_LINEAR: return byM(Mc, std::integral_constant<int, F_LINEAR>{});
            case F_DMT: return byM(Mc, std::integral_constant<int, F_DMT>{});
            case F_DMT_KV: return byM(Mc, std::integral_constant<int, F_DMT_KV>{});
            case F_HOOKE: return byM(Mc, std::integral_constant<int, F_HOOKE>{});
            case F_SPRING_DAMPER: return byM(Mc, std::integral_constant<int, F_SPRING_DAMPER>{});
        }
        return cudaErrorInvalidValue;
    };
    if (K.m == 1) return byF(std::integral_constant<int, 1>{});
    if (K.m == 3) return byF(std::integral_constant<int, 3>{});
    return byF(std::integral_constant<int, AFM_MAXM>{});
}

}  // namespace afm
