// afm_launch.h -- host-side launchers of the CUDA kernels (C++ linkage,
// internal to libafminv).  Each returns the cudaError_t of its launch.
#pragma once
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include "../../include/afminv.h"
#include "afm_internal.h"

namespace afm {

struct SwarmPtrs {
    float* x;                  // [D][P]
    float* v;                  // [D][P]
    float* pb[2];              // personal-best positions, double-buffered by iteration parity
    float* pbS;                // [P]
    unsigned long long* gkey[2];  // global-best key words (S bits << 32 | particle), by parity
    int* flags;                // [1] non-finite counter
};

struct PsoConst {
    int P, D, iters;
    float w, c1, c2;
    uint64_t seed;
    uint32_t pixel;
    uint32_t p0;   // swarm-wide index of particle 0 (a slice of a split swarm; else 0)
};

// forward + optional misfit; lanes (afm_lanes): AFM_LANES_ONE keeps one
// particle per thread, any other value pairs particles in paired FP32
// instructions for large DMT batches (1 or 3 modes, P >= 65 536;
// bit-identical)
cudaError_t launch_forward_f32(const KConst<float>& K, const float* x, int P, float* defl,
                               const float* U, float* S, int* flags, cudaStream_t st,
                               int lanes = 0);
cudaError_t launch_forward_f64(const KAffine<double>& K, const double* x, int P, double* defl,
                               const double* U, double* S, int* flags, cudaStream_t st);
// standalone misfit of a time-major deflection array
cudaError_t launch_misfit(const float* defl, const float* U, int N, int P, float* S, int num_sms,
                          cudaStream_t st);
// synthetic records: FP32 at the fine step of K, sampled every `sub`, plus noise
cudaError_t launch_synth(const KConst<float>& K, const double* x_truth, int n_pix,
                         const int64_t* off, int sub, float sigma_nm, uint64_t seed,
                         uint32_t pixel0, float* U_cat, cudaStream_t st);

// Per-pixel problem constants of a batch whose pixels differ in their
// cantilever or set-point (afm_problem per pixel): indexed by pixel id, with
// each pixel's drive g at its 2 spc half-step phases (+ wrap entry) in FP32
// and the drive terms of the affine step: FP32 rows and the FP64 sine and
// cosine of each phase (tab64).  kf == nullptr: every pixel uses the launch's constants.
struct PixConst {
    const KAffine<float>* kf;   // [n_pix]
    const KAffine<double>* kd;  // [n_pix]
    const double* tab64;        // [n_pix][ld64]
    const float* tab32;         // [n_pix][ld]
    const float* rows;          // [n_pix][ld_rows]
    int ld, ld64, ld_rows;
};
// fills the tables of n_pix pixels from kd and kf
cudaError_t launch_pix_tables(const PixConst& pc, int m, int force, int n_pix, int spc2,
                              cudaStream_t st);

// many independent pixel inversions in one persistent launch
struct BatchArgs {
    const float* U;        // concatenated records
    const int64_t* off;    // [n_pix + 1]
    const int* order;      // queue order of pixels (longest first) or nullptr
    int n_pix;
    uint32_t pixel0;       // Philox counter word 2 of pixel 0
    int* queue;            // batch_queue_words(n_pix) words, zeroed before the launch
    int layer;             // > 0: a block per pixel on `layer` SMs, dealt by batch_deal;
                           // 0: blocks pull pixels until the queue is empty
    afm_result* res;       // [n_pix]
    float* pb_out;         // nullptr, or per queue slot the final personal bests
                           // [D][P] (normalised cube) followed by their misfits [P]
    // optional prior per queue slot (image scans): the swarm searches the box
    // [box_lo, box_hi] ([slot][D], normalised) in box-local coordinates, and
    // particles p < n_seed start at seeds [slot][n_seed][D]
    const float* box_lo;
    const float* box_hi;
    const float* seeds;
    int n_seed;
    PixConst pix;          // per-pixel constants (pix.kf == nullptr: shared)
};
// Where every pixel has a resident block, slots (longest first) are dealt to
// the SMs in layers of one slot per SM, to and fro, the last full layer
// longest last: the SMs' sums are even or, where a rest follows, smaller on
// the SMs that get one of it.  SM i's slot of layer l:
__host__ __device__ inline int batch_deal(int l, int i, int n, int sms) {
    const int full = n / sms;
    return l * sms + (l < full && (full - l) % 2 ? sms - 1 - i : i);
}
// Words of BatchArgs::queue: counters, per SM (id modulo 256) its blocks and
// its index, and for a dealt launch a flag per slot.
constexpr int BATCH_SMS = 256, BATCH_FLAGS = 4 + 2 * BATCH_SMS;
inline size_t batch_queue_words(int n_pix) { return (size_t)BATCH_FLAGS + (size_t)n_pix; }
int batch_threads(int P, int kp);
// largest block of the batch kernel with kp particles per thread (the
// paired-instruction kernels of kp = 2, 4 are built for up to 128 registers)
int batch_max_threads(int kp);
// dynamic shared memory of the batch kernel (pp: per-pixel constants)
size_t batch_smem(int P, int D, int spc2, bool pp = false);
int batch_sort_max();
cudaError_t batch_sort(const int64_t* off, int n_pix, int* order, cudaStream_t st);
cudaError_t batch_occupancy(int m, int force, int kp, int P, int D, int spc2, bool pp,
                            int* blocks_per_sm);
cudaError_t launch_batch(const KConst<float>& K, const PsoConst& pc, const BatchArgs& a, int kp,
                         int grid, cudaStream_t st);

// discrete adjoint (gradient of the misfit wrt the normalised parameters)
// Ragged form (off != nullptr): particle p belongs to queue slot p / per_slot,
// pixel order[slot] (or the slot itself), and is compared with that pixel's
// record U + off[pix] of length off[pix+1] - off[pix] <= K.n_steps; records
// longer than K.n_steps give S = inf and a zero gradient.
size_t adjoint_ckpt_floats(int m, int n_steps, int P);
// One record for all particles, its segments at once (kern_adjoint.cu): for
// batches and workspaces that adjoint_runs_split accepts; adjoint_ws_floats has
// room for it wherever it pays.
bool adjoint_runs_split(int m, int force, int n_steps, int spc, int P, const void* ws,
                        size_t ws_bytes);
cudaError_t launch_adjoint_split(const KAffine<float>& K, const float* x, int P, const float* U,
                                 float* S, float* G, float* ws, cudaStream_t st);
size_t adjoint_ws_floats(int m, int force, int n_steps, int P);
cudaError_t launch_adjoint(const KConst<float>& K, const float* x, int P, const float* U, float* S,
                           float* G, float* ckpt, cudaStream_t st, const int64_t* off = nullptr,
                           const int* order = nullptr, int per_slot = 1);

// Levenberg-Marquardt polish (kern_lm.cu): sensitivity pass (S [P], H
// [P][D][D], b [P][D]; ragged form as launch_adjoint), damped trial points,
// choice of the best trial point
// (pix: per-pixel constants of the ragged form, pix.kf == nullptr: K for all)
cudaError_t launch_sens(const KAffine<float>& K, const float* x, int P, const float* U, float* S,
                        double* H, double* b, cudaStream_t st, const int64_t* off = nullptr,
                        const int* order = nullptr, int per_slot = 1,
                        const PixConst& pix = PixConst{});
// the same pass with one lane per parameter direction (kern_lm_lanes.cu);
// launch_sens uses it when P x lanes fits one warp per SM sub-partition
bool sens_lanes_preferred(int P, int D);
cudaError_t launch_sens_lanes(const KAffine<float>& K, const float* x, int P, const float* U,
                              float* S, double* H, double* b, cudaStream_t st, const int64_t* off,
                              const int* order, int per_slot);
cudaError_t launch_lm_cand(int D, int K, int J, const float* x, const double* H, const double* b,
                           double lam0, double ratio, float* Xc, cudaStream_t st);
cudaError_t launch_lm_select(int D, int K, int J, float* x, float* S, const float* Xc,
                             const float* Sc, cudaStream_t st);
// the choice of the fused step (trial points through the sensitivity pass):
// the point kept brings its H [D][D] and b [D] from Hc [K*J][D][D], bc [K*J][D]
cudaError_t launch_lm_select_hb(int D, int K, int J, float* x, float* S, double* H, double* b,
                                const float* Xc, const float* Sc, const double* Hc,
                                const double* bc, cudaStream_t st);

// image scans (kern_image.cu): coarse and fine pixel lists of a row-major
// width x height image with coarse spacing `stride`; per fine pixel a box
// around its (up to 4) coarse neighbours' winners, widened by `margin`, and
// those winners as 4 seed points
void image_counts(int width, int height, int stride, int* n_coarse, int* n_fine);
cudaError_t launch_image_plan(int width, int height, int stride, int* coarse, int* fine,
                              cudaStream_t st);
cudaError_t launch_image_prior(int width, int height, int stride, int D, float margin,
                               const afm_result* res, const int* fine, int n_fine, float* box_lo,
                               float* box_hi, float* seeds, cudaStream_t st);

// batched polish (kern_bpolish.cu): candidates of queue slot s are columns
// s * Kc .. s * Kc + Kc - 1 of [D][n_pix * Kc] arrays
cudaError_t launch_topk_pix(const float* pb_all, int n_pix, int P, int D, int Kc, float* xk,
                            float* Sk, int* ik, cudaStream_t st);
cudaError_t launch_forward_ragged(const KConst<float>& K, const float* x, int Ptot, const float* U_cat,
                                  const int64_t* off, const int* order, int per_slot, float* S,
                                  cudaStream_t st, const PixConst& pix = PixConst{});
cudaError_t launch_pick_pix(int n_pix, int D, int Kc, const float* xk, const float* Sk,
                            const int* ik, const int* order, int iters, afm_result* res,
                            cudaStream_t st);

// gradient polish
cudaError_t launch_polish_cand(int D, int K, int J, const float* x, const float* G, double alpha0,
                               double shrink, float* Xc, cudaStream_t st);
cudaError_t launch_polish_select(int D, int K, int J, float sigma, float* x, const float* G,
                                 float* S, const float* Xc, const float* Sc, cudaStream_t st);
cudaError_t launch_topk(const float* pbS, const float* pb, int P, int D, int K, float* xk, int* idx,
                        cudaStream_t st);
cudaError_t launch_polish_final(const KConst<double>& K, int Kn, int iters, const float* x,
                                const float* S, const int* idx, const float* U, const int* flags,
                                void* result, cudaStream_t st);

// finite-element cantilever
cudaError_t launch_fe_forward_f32(const FeConst& F, const float* x, int P, float* defl,
                                  const float* U, float* S, cudaStream_t st);
cudaError_t launch_fe_forward_f64(const FeConst& F, const double* x, int P, double* defl,
                                  const double* U, double* S, cudaStream_t st);
cudaError_t launch_fe_invert_iter(const FeConst& F, const PsoConst& pc, const SwarmPtrs& sw,
                                  const float* U, float* history, int it, cudaStream_t st);
cudaError_t launch_fe_invert_final(const FeConst& F, const PsoConst& pc, const SwarmPtrs& sw,
                                   const float* U, float* history, void* result, cudaStream_t st);

// particle swarm
cudaError_t launch_pso_init(const PsoConst& pc, const SwarmPtrs& sw, cudaStream_t st);
cudaError_t launch_pso_best(const PsoConst& pc, const SwarmPtrs& sw, const float* S, int it,
                            cudaStream_t st);
cudaError_t launch_pso_move(const PsoConst& pc, const SwarmPtrs& sw, int it, cudaStream_t st);
// the move with a given global-best position gb [D] (a slice of a split swarm)
cudaError_t launch_pso_move_given(const PsoConst& pc, const SwarmPtrs& sw, const float* gb, int it,
                                  cudaStream_t st);
// fused inversion iteration (it = 0: initial evaluation)
cudaError_t launch_invert_iter(const KConst<float>& K, const PsoConst& pc, const SwarmPtrs& sw,
                               const float* U, float* history, int it, cudaStream_t st);
// base-motion inversion (drive_mode 1, kern_drive.cu)
cudaError_t launch_forward_drive_f32(const KConst<float>& K, const float* x, int P, float* defl,
                                     const float* U, float* S, cudaStream_t st);
cudaError_t launch_forward_drive_f64(const KConst<double>& K, const double* x, int P, double* defl,
                                     const double* U, double* S, cudaStream_t st);
cudaError_t launch_invert_drive(const KConst<float>& K, const PsoConst& pc, const SwarmPtrs& sw,
                                const float* U, float* history, int it, cudaStream_t st);
cudaError_t launch_drive_final(const KConst<double>& K, const PsoConst& pc, const SwarmPtrs& sw,
                               const float* U, float* history, void* result, cudaStream_t st);
// deflections at several points along the cantilever (n_points > 0, kern_points.cu)
cudaError_t launch_forward_points_f32(const KConst<float>& K, const float* x, int P, float* defl,
                                      const float* U, float* S, cudaStream_t st);
cudaError_t launch_forward_points_f64(const KConst<double>& K, const double* x, int P, double* defl,
                                      const double* U, double* S, cudaStream_t st);
cudaError_t launch_invert_points(const KConst<float>& K, const PsoConst& pc, const SwarmPtrs& sw,
                                 const float* U, float* history, int it, cudaStream_t st);
cudaError_t launch_points_final(const KConst<double>& K, const PsoConst& pc, const SwarmPtrs& sw,
                                const float* U, float* history, void* result, cudaStream_t st);
// winner re-evaluation in FP64 and result record
cudaError_t launch_invert_final(const KConst<double>& K, const PsoConst& pc, const SwarmPtrs& sw,
                                const float* U, float* history, void* result, cudaStream_t st);

// FP64 re-evaluation of one winner by multiple shooting in time
// (kern_reeval.cu): segments of AFM_SEG steps, B = ceil(n_steps / AFM_SEG).
struct ReevalWinner {
    double x[AFM_MAXD];   // normalised parameters
    double c[4];          // FP64 force coefficients (written by the guess kernel)
    float S32;            // FP32 misfit that selected the winner
    int winner;           // its particle index
};
struct ReevalPtrs {
    ReevalWinner* win;
    double* tab;          // [2 spc] sine and cosine of the phases (room for spc2 + 1)
    double* start[2];     // [B + 1][2m] segment start states (alternating sweeps)
    double* E;            // [B][2m] segment end states
    double* J;            // [B][2m][2m] segment tangent maps
    double* Sb;           // [B] segment misfit shares
    double* sumU2;        // [1]
    int B;
};
// The same for every queue slot of a batch (kern_reeval_batch.cu): slot i
// owns segments [i maxB, (i + 1) maxB) of the segment arrays.
struct ReevalBatch {
    double* coef;   // [n_pix][4] FP64 force coefficients of each slot's winner
    double* tab;    // FP64 drive terms of every phase (aff::Table)
    double* Z;      // [n_pix * maxB][2m] segment start states (corrected in place)
    double* E;      // [n_pix * maxB][2m] segment end states
    float* J;       // [n_pix * maxB][2m][2m] segment tangent maps (FP32)
    double* Sb;     // [n_pix * maxB] segment misfit shares
    double* u2;     // [n_pix] sum of U^2 of each slot's record
    int maxB;       // segments of the longest record (problem n_steps)
};
size_t reeval_batch_bytes(int m, int force, int n_steps, int spc, int n_pix);
void reeval_batch_carve(void* base, int m, int force, int n_steps, int spc, int n_pix,
                        ReevalBatch* R);
// fills each slot's result record (S_f64, J_rel, theta, status, defect,
// segments) from the parameters already in it
cudaError_t launch_reeval_batch(const KAffine<float>& Kf, const KAffine<double>& Kd,
                                const ReevalBatch& R, const BatchArgs& a, cudaStream_t st);
bool reeval_supported(int m, int n_steps);
size_t reeval_bytes(int m, int n_steps, int spc);
void reeval_carve(void* base, int m, int n_steps, int spc, ReevalPtrs* R);
cudaError_t launch_reeval_pick_swarm(const PsoConst& pc, const SwarmPtrs& sw, float* history,
                                     ReevalWinner* w, cudaStream_t st);
cudaError_t launch_reeval_pick_min(int D, int Kn, const float* x, const float* S, const int* idx,
                                   ReevalWinner* w, cudaStream_t st);
cudaError_t launch_reeval(const KAffine<float>& Kf, const KAffine<double>& Kd, const ReevalPtrs& R,
                          const float* U, int iters, const int* flags, void* result,
                          cudaStream_t st);

}  // namespace afm
