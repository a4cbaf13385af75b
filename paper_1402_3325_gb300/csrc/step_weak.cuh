// step_weak.cuh -- the pair kernels that solve weakly perturbed pairs with
// kepler_weak.cuh: launchers.
#pragma once

#include "step_grp.cuh"
#include "step_common.cuh"

namespace sakura {

// rows [4][n] of the particles as the weak pair kernels read them
// (kepler_weak.cuh), written by the prep kernel and the fused apply kernels
struct WeakStep {
    float4 *rows;
    double inv_t;  // 1 / tau
};

// The forms that have weak kernels: FP64 with the single-precision seed,
// double-word (no float copy X32), mixed under the literal rule with e_max < 1
// and the seed (StepArgs rule, post32), FP64 with an analytic or the learned
// guess (no X32, no statistics).
enum class WeakForm { Fp64, Df64, Mixed, Guess, Learned };

// The choice of a run's kernels, by the prep kernel from sampled pairs of the
// state: p->every = 0 those of the weak pairs, 1 those that solve every pair
// (more than limit of kWeakSample pairs strong; unbound: weak pairs are
// unbound ones only, the mixed form's rule).
constexpr int kWeakSample = 1024;
struct WeakChosen {
    int every;
    unsigned sum;  // of the sample's blocks; zero between runs
};
struct WeakChoice {
    WeakChosen *p;
    int limit;
    bool unbound;
    float *X3;  // three-float copy that the prep kernel writes (double-word form) or null
};

void launch_prep_weak(const double *state, const double *mass, double *X, float *X32,
                      float4 *rows, int64_t n, double tau, unsigned *status, const WeakChoice &ch,
                      cudaStream_t s);
void launch_pair_step_weak(const StepArgs &a, const WeakStep &ws, int Smax, int64_t T, int blocks,
                           bool stats, WeakForm form, cudaStream_t s);
int pair_step_weak_blocks_per_sm(bool stats, WeakForm form);
void launch_pair_step_grp_weak(const StepArgs &a, const WeakStep &ws, const GrpLayout &L,
                               const GrpParts &parts, int blocks, bool stats, WeakForm form,
                               cudaStream_t s);
int pair_step_grp_weak_blocks_per_sm(bool stats, WeakForm form);

// The small kernel: the state and the masses before the step, and the
// tile-steps of a warp (2, 4 or 8; a block takes four times as many, the grid
// 32 / (4 steps) blocks per tile).
struct WeakSmall {
    const double *src, *mass;
    double inv_t;  // 1 / tau
    int steps;
};

// three: room for three blocks per SM instead of two
void launch_pair_step_weak_small(const StepArgs &a, const WeakSmall &ws, int blocks, bool three,
                                 bool stats, WeakForm form, cudaStream_t s);
void launch_apply_weak_small(const double *src, double *dst, const double *partial, int n,
                             int slots, double tau, unsigned *status, cudaStream_t s);
void launch_copy_state(const double *src, const double *mass, double *dst, double *mdst, int n,
                       cudaStream_t s);

}  // namespace sakura
