// afm_internal.h -- structures shared by the host set-up (afminv_api.cpp) and
// the CUDA kernels.  Not part of the public ABI.
//
// Units inside the kernels ("scaled units"):
//   length  1 nm
//   time    tau = h / 6, where h = 1 / (f1 * steps_per_cycle) is the RK4 step,
//           so that the RK4 constants h/2 = 3, h = 6 and h/6 = 1 are exact
//           binary numbers (an FP32 rounding of h/6 would detune the resonant
//           mode against the index-exact drive by ~3e-8 per step, which a
//           quality factor of 400 amplifies to ~6e-6 of the deflection)
//   force   k * 1 nm * (omega_1 tau)^2, so the modal equation (Eq. 2) reads
//             q_i'' = tip_i F + gamma_i g - w2_i q_i - wq_i q_i'
//           with w2_i = (omega_i tau)^2, wq_i = omega_i tau / Q_i.
#pragma once
#include <stdint.h>

#define AFM_MAXM 8
#define AFM_MAXD 5
#define AFM_TAB_MAX 4096   // half-step drive phases per period (2 * steps_per_cycle)
#define AFM_SEG 32         // adjoint checkpoint interval (RK4 steps)

#if defined(__CUDACC__)
#define AFM_HD __host__ __device__
#else
#define AFM_HD
#endif

namespace afm {

// Which modes take compensated (Kahan) state updates.  FP64: all.  FP32: the
// lowest mode only.  It carries the resonant response, and its RK4 increment
// is a small fraction of the state (omega_1 h << 1), so that a plain sum
// drops low bits of the deflection every step; the higher modes are driven
// far off resonance, with amplitudes ~(omega_1 / omega_i)^2 / Q of the first
// mode's, and their plain-sum rounding stays far below FP32 resolution of
// the tip deflection.
template <typename T>
AFM_HD constexpr bool comp_mode(int i) {
    return sizeof(T) == 8 || i == 0;
}

enum ForceKind { F_LINEAR = 0, F_DMT = 1, F_DMT_KV = 2, F_HOOKE = 3, F_SPRING_DAMPER = 4 };

// Force-law coefficients of one particle in scaled units.
//   LINEAR        F = -c0 (d - c1)
//   DMT           F = c0 max(c3 - d, 0)^1.5 - c1 / max(d, c3)^2      (c0 = hz, c1 = vdw, c3 = a0)
//   DMT_KV        DMT - c2 sqrt(max(c3 - d, 0)) d'                    (c2 = kv)
//   HOOKE         F = c0 max(c1 - d, 0)
//   SPRING_DAMPER F = (d < c1) ? c0 (c1 - d) - c2 d' : 0
template <typename T>
struct Coef {
    T c0, c1, c2, c3;
};

// The RK4 step of the modal cantilever as an affine map (host set-up:
// affine_setup).  Between the four tip forces F1..F4 of a step everything is
// linear, so the stage gaps and the step's increments are fixed combinations
// of the state, the earlier stage forces and drive terms that depend only on
// the phase: the classic stages (Eq. 2, Sec. 3.2) with the algebra done once
// per problem in FP64 instead of once per step in the kernel.
//
// State per mode: the deflection q and a second coordinate,
//   mode 0   w = B v + A1 q, the part of the step's increment of q that is
//            linear in the state: q' - q = w + (forces, drive), and
//            w' - w = c (q + w) + ec w + ...; ec = det - 1 alone carries the
//            damping and c (with a low word) the frequency of the resonant
//            mode, so that FP32 coefficients keep both to ~1e-8 relative
//   others   p = 3 v (robust at any omega h; mode 0's form is singular where
//            B = 0), with A1, B, C, D1 of the 2 x 2 step matrix rounded
//            together so that its frequency and damping keep ~1e-9
// Stage gaps: d1 = zq + s1, d2 = zq + (s1 + ...), with zq = Zc + q_0 and
// the small remainders summed first; d3, d4 add e31 F1 and e41 F1 + e42 F2.
#define AFM_AFF_TAB 24   // drive terms per phase, at most (8 modes, rate law: 21)
template <typename T>
struct Affine {
    T d2q, d2w;                              // stage 2 of mode 0 beyond q_0
    T d3q[AFM_MAXM], d3p[AFM_MAXM];          // stage 3, 4 gaps (mode 0: beyond q_0)
    T d4q[AFM_MAXM], d4p[AFM_MAXM];
    T e31, e41, e42;
    T ec, c0, c0lo;                          // mode 0's second coordinate
    T A1[AFM_MAXM], B[AFM_MAXM], C[AFM_MAXM], D1[AFM_MAXM];   // modes >= 1
    T bq[3][AFM_MAXM], bp[4][AFM_MAXM];      // increments per unit stage force
    // gap rates of the stages (laws with a rate term); stage 1:
    // v1q q_0 + v1w w_0 + (sum of p_i) / 3
    T v1q, v1w, third;
    T r2q[AFM_MAXM], r2p[AFM_MAXM], r3q[AFM_MAXM], r3p[AFM_MAXM], r4q[AFM_MAXM], r4p[AFM_MAXM];
    T h21, h31, h32, h41, h42, h43;
    T p0[AFM_MAXM];                          // initial second coordinates
    // drive term k at phase j: dS[k] sin(2 pi j / spc) + dC[k] cos(2 pi j / spc);
    // k = 0, 1: gaps of stages 3, 4; 2 + i, 2 + M + i: increments of q_i and
    // of the second coordinate (M: the kernels' template mode count);
    // 2 + 2 M ..: gap rates of stages 2, 3, 4
    double dS[AFM_AFF_TAB], dC[AFM_AFF_TAB];
};

// Template mode count of the kernels for m modes (modes past m have zero
// constants), and the words per phase of their drive-term rows.
AFM_HD constexpr int aff_modes(int m) { return (m == 1 || m == 3) ? m : AFM_MAXM; }
AFM_HD constexpr int aff_row(int M, bool rate) { return (2 + 2 * M + (rate ? 3 : 0) + 3) & ~3; }
// words per phase of an FP64 table (aff::Table<double>)
AFM_HD constexpr int aff_row64(int M, bool rate) { return M > 3 ? 2 : aff_row(M, rate); }
AFM_HD constexpr bool rate_law(int force) { return force == 2 || force == 4; }

// Constants of one problem in the arithmetic type of a kernel (float or
// double), filled on the host by the per-problem set-up.
template <typename T>
struct KConst {
    // The arrays start 8 bytes past a 16-byte boundary, here and in KAffine: on
    // one, the compiler reads them 16 bytes at a time into more registers, and
    // the eight-mode kernels were slower (DMT, 19 457 particles x 512 steps 220
    // us, 211 so; Hooke's sensitivities, 512 x 512 steps, 212 us, 196 so).  The
    // batch kernel's copy in shared memory has them on one.
    double skew;
    T w2[AFM_MAXM], w2lo[AFM_MAXM], wq[AFM_MAXM], gam[AFM_MAXM], tip[AFM_MAXM];
    T q0[AFM_MAXM], v0[AFM_MAXM];
    T Zc;
    double drive_amp, drive_phase;  // g = drive_amp * sin(2 pi j / spc2 + drive_phase)
    int m, spc2, n_steps, force, D;
    int slot[AFM_MAXD], logs[AFM_MAXD];
    double lo[AFM_MAXD], span[AFM_MAXD], fixed[AFM_MAXD];
    double k, s1, tau;
    int drive_mode;                 // 1: per-particle base motion from rest (kern_drive.cu)
    double drv[3];                  // fixed base amplitude [m], frequency [Hz], chirp [Hz/s]
    int np;                         // deflection points (kern_points.cu), 0: the tip
    T phi[4][AFM_MAXM];             // tip-normalised mode shapes at the points
};

// The constants with the step's affine map, for the kernels that run it.  The
// stage-form kernels (every FP32 solve and swarm) take KConst alone: the map is
// two thirds of the words, and forming it costs the host 2 of a call's 11 us for
// three modes in FP32, 6 of 22 for eight (10 and 30 us on an x86 core), once per
// pixel where the pixels' problems differ.
template <typename T>
struct AffineFirst {
    Affine<T> af;
    double skew[3];   // see KConst
};
template <typename T>
struct KAffine : AffineFirst<T>, KConst<T> {};
// no padding between or after: the bytes are part of a launch graph's key
static_assert(sizeof(KAffine<float>) == sizeof(KConst<float>) + sizeof(Affine<float>) + 24 &&
                  sizeof(KAffine<double>) == sizeof(KConst<double>) + sizeof(Affine<double>) + 24,
              "KAffine has padding");

// Finite-element cantilever (cubic Hermite elements, clamped node removed)
// advanced by Newmark's average-acceleration scheme (beta = 1/4, gamma = 1/2)
// with the tip force implicit.  With Rayleigh damping, M, K and C are
// diagonal in the M-orthonormal eigenbasis (u = Phi z, Phi^T M Phi = I), so
// the scheme decouples exactly into one scalar recursion per mode, written in
// increment form (delta = z_n - z_{n-1}):
//   delta_{n+1} = delta_n + b1_i z_n + d2_i delta_n + g_i G_n
//                 + f_i (F_{n+1} + 2 F_n + F_{n-1}),   z_{n+1} = z_n + delta_{n+1}
// with s_i = 1 + h/2 c_i + h^2/4 lambda_i, b1_i = -h^2 lambda_i / s_i,
// d2_i = -h c_i / s_i (c_i = alpha + beta lambda_i), g_i = (phi_i^T M r) / s_i
// (G_n = table_{n+1} + 2 table_n + table_{n-1}, table = h^2/4 g in nm) and
// f_i = (h^2/4) k phi_i(tip) / s_i (force in units of k * 1 nm); the tip
// deflection is sum_i phi_i(tip) z_i.
#define AFM_FE_MAXN 64      // DOFs = modes (2 per node)
#define AFM_FE_LANES 8      // lowest modes with compensated sums in FP32 (the 8-lane layout's slot 0)

struct FeConst {
    int ne, n, spc, n_steps;
    double h;                   // Newmark step (s)
    double Zc;                  // rest gap [nm]
    double drive_amp, drive_phase;   // table_j = drive_amp sin(2 pi j / spc + phase)
    double b1[AFM_FE_MAXN], d2[AFM_FE_MAXN], g[AFM_FE_MAXN], f[AFM_FE_MAXN], pt[AFM_FE_MAXN];
    // b1 of the lowest AFM_FE_LANES modes carries a low word in FP32 (the
    // resonant mode's frequency must be represented to ~1e-12)
    double z0[AFM_FE_MAXN], dz0[AFM_FE_MAXN];   // initial modal state and increment
    double ctip;                // sum_i pt_i f_i: tip response to the step's own tip force
    double utip0, utipm;        // tip deflection at steps 0 and -1 [nm]
    KConst<float> pm;           // force law and parameter map (s1 = 1)
};

}  // namespace afm
