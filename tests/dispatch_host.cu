// Launchers of csrc/sakura_api.cu's kernels that launch nothing, for
// tests/test_dispatch_host.py: each notes its name and whether what its kernel
// would read lies in scratch that the library still holds
// (tests/dispatch_runtime.cpp).
#include <cstring>
#include <vector>

#include "../paper_1402_3325_gb300/csrc/mlp_infer.cuh"
#include "../paper_1402_3325_gb300/csrc/step_batched.cuh"
#include "../paper_1402_3325_gb300/csrc/step_common.cuh"
#include "../paper_1402_3325_gb300/csrc/step_grp.cuh"
#include "../paper_1402_3325_gb300/csrc/step_small.cuh"
#include "../paper_1402_3325_gb300/csrc/step_weak.cuh"

bool held(const void *p, size_t bytes);
void note(const char *name, bool ok);

namespace sakura {

namespace {
size_t doubles(int64_t k) { return (size_t)k * sizeof(double); }

bool state_ok(const double *src, const double *mass, const double *X, int64_t n)
{
    return held(src, doubles(6 * n)) && held(mass, doubles(n)) && held(X, doubles(7 * n));
}
}  // namespace

void launch_prep_weak(const double *src, const double *mass, double *X, float *X32, float4 *rows,
                      int64_t n, double, unsigned *, const WeakChoice &ch, cudaStream_t)
{
    note("prep_weak", held(ch.p, sizeof(*ch.p)) &&
                          (!ch.X3 || held(ch.X3, 80 * (size_t)n)) && state_ok(src, mass, X, n) && (size_t)rows % 16 == 0 &&
                          held(rows, 64 * (size_t)n) && (!X32 || held(X32, 40 * (size_t)n)));
    std::memcpy(X + 6 * n, mass, doubles(n));
}
void launch_prep_step(const double *src, const double *mass, double *X, float *X32, int64_t n,
                      double, unsigned *, cudaStream_t)
{
    note("prep", state_ok(src, mass, X, n) && (!X32 || held(X32, 40 * (size_t)n)));
    std::memcpy(X + 6 * n, mass, doubles(n));
}
void launch_prep_mixed(const double *src, const double *mass, double *X, float *X32, int64_t n,
                       double, unsigned *, cudaStream_t)
{
    note("prep_mixed", state_ok(src, mass, X, n) && held(X32, 40 * (size_t)n));
}
void launch_prep_df64(const double *src, const double *mass, double *X, float *X3, int64_t n,
                      double, unsigned *, cudaStream_t)
{
    note("prep_df64", state_ok(src, mass, X, n) && held(X3, 80 * (size_t)n));
}
void launch_copy_state(const double *src, const double *mass, double *dst, double *mdst, int n,
                       cudaStream_t)
{
    note("copy", held(src, doubles(6 * n)) && held(mass, doubles(n)) &&
                     held(dst, doubles(6 * n)) && held(mdst, doubles(n)));
}

namespace {
bool args_ok(const StepArgs &a)
{
    return held(a.X, doubles(7 * a.n)) && (!a.X32 || held(a.X32, 40 * (size_t)a.n)) &&
           (!a.gate.p || held(a.gate.p, sizeof(int)));
}

// a weak step's other set of kernels, which solves every pair: "every_..."
void note_pairs(const char *name, const StepArgs &a, bool ok)
{
    static char every[32];
    std::strcat(std::strcpy(every, "every_"), name);
    note(a.gate.p && a.gate.open == 1 ? every : name, ok);
}

// the tiles' partial sums
bool slots_ok(const StepArgs &a, int Smax)
{
    return held(a.partial, doubles((a.n + 31) / 32 * Smax * 6 * a.n));
}
}  // namespace

void launch_pair_step_weak(const StepArgs &a, const WeakStep &ws, int Smax, int64_t, int, bool,
                           WeakForm, cudaStream_t)
{
    note("weak", args_ok(a) && slots_ok(a, Smax) && a.gate.p && held(ws.rows, 64 * (size_t)a.n));
}
void launch_pair_step_grp_weak(const StepArgs &a, const WeakStep &ws, const GrpLayout &,
                               const GrpParts &parts, int blocks, bool, WeakForm, cudaStream_t)
{
    note("grp_weak", args_ok(a) && a.gate.p && held(ws.rows, 64 * (size_t)a.n) &&
                         held(parts.colx, doubles(192 * (int64_t)blocks)));
}
void launch_pair_step_weak_small(const StepArgs &a, const WeakSmall &ws, int, bool, bool, WeakForm,
                                 cudaStream_t)
{
    const int64_t nb = (a.n + 31) / 32;
    note("small_weak", held(ws.src, doubles(6 * a.n)) && held(ws.mass, doubles(a.n)) &&
                           held(a.partial, doubles(nb * (8 / ws.steps) * 6 * a.n)));
}
void launch_apply_weak_small(const double *src, double *dst, const double *, int n, int, double,
                             unsigned *, cudaStream_t)
{
    note("small_apply", held(src, doubles(6 * n)) && held(dst, doubles(6 * n)));
}
void launch_pair_step_sym(const StepArgs &a, int Smax, int64_t, int, bool, cudaStream_t)
{
    note_pairs("sym", a, args_ok(a) && slots_ok(a, Smax));
}
void launch_pair_step_df64(const StepArgs &a, const DwArgs &da, int Smax, int64_t, int, bool,
                           cudaStream_t)
{
    note_pairs("df64", a, args_ok(a) && slots_ok(a, Smax) && held(da.X3, 80 * (size_t)a.n));
}
void launch_pair_step_fp64(const StepArgs &a, int, int, bool, cudaStream_t)
{
    note("ordered", args_ok(a));
}
void launch_pair_step_mixed(const StepArgs &a, const MixedArgs &, int, bool, cudaStream_t)
{
    note("ordered_mixed", args_ok(a));
}
void launch_pair_step_grp(const StepArgs &a, const GrpLayout &, const GrpParts &parts, int blocks,
                          bool, cudaStream_t)
{
    note_pairs("grp", a, args_ok(a) && held(parts.colx, doubles(192 * (int64_t)blocks)));
}
void launch_pair_step_grp_mixed(const StepArgs &a, const MixedArgs &, const GrpLayout &,
                                const GrpParts &, int, bool, cudaStream_t)
{
    note("grp_mixed", args_ok(a));
}
void launch_pair_step_grp_df64(const StepArgs &a, const DwArgs &da, const GrpLayout &,
                               const GrpParts &parts, int blocks, bool, cudaStream_t)
{
    note_pairs("grp_df64", a, args_ok(a) && held(da.X3, 80 * (size_t)a.n) && held(parts.colx, doubles(192 * (int64_t)blocks)));
}
void launch_apply_sym(double *dst, double *X, float *, float4 *rows, const double *, int64_t n, int,
                      int64_t, int64_t, double, bool, double, unsigned *, const SymAlt &alt,
                      cudaStream_t)
{
    note("apply_sym", (!alt.X3 || held(alt.X3, 80 * (size_t)n)) &&
                      held(dst, doubles(6 * n)) && held(X, doubles(7 * n)) &&
                          (!rows || held(rows, 64 * (size_t)n)));
}
void launch_apply_grp(double *dst, double *X, float *, float4 *rows, const GrpParts &, int64_t n,
                      const GrpLayout &, int64_t, double, bool, double, unsigned *,
                      const GrpAlt &alt, cudaStream_t)
{
    note("apply_grp", (!alt.X3 || held(alt.X3, 80 * (size_t)n)) && held(dst, doubles(6 * n)) && held(X, doubles(7 * n)) &&
                          (!rows || held(rows, 64 * (size_t)n)));
}
void launch_apply_df64(double *dst, const double *X, const void *, int64_t n, int, int64_t, int64_t,
                       double, unsigned *, cudaStream_t)
{
    note("apply_df64", held(dst, doubles(6 * n)) && held(X, doubles(7 * n)));
}
void launch_apply_step(double *dst, const double *X, const double *, int64_t n, int64_t, double,
                       unsigned *, cudaStream_t)
{
    note("apply", held(dst, doubles(6 * n)) && held(X, doubles(7 * n)));
}
void launch_small(const SmallArgs &, bool, bool, bool, cudaStream_t) { note("single_block", true); }
void launch_energy(const double *, const double *, int64_t, double *, double *, unsigned *,
                   unsigned *, cudaStream_t)
{
}
void launch_batched(const BatchArgs &, int, int, bool, cudaStream_t) {}
cudaError_t build_batched_graph(const BatchArgs &, int, int, bool, cudaGraphExec_t *)
{
    return cudaErrorNotSupported;
}
void build_batch_schedule(const int64_t *, int, std::vector<int> &, std::vector<int> &) {}
void launch_pair_classes(const float *, int64_t, const ClassRule &, unsigned char *, cudaStream_t) {}
void launch_sample_pairs(const double *, int64_t, double, double, const int64_t *, int64_t, float *,
                         float *, int *, double, unsigned *, cudaStream_t)
{
}
void launch_mlp_eval(const MlpWeights *, const float *, int64_t, float *, cudaStream_t) {}
void launch_mlp_pack(const float *, MlpWeights *, cudaStream_t) {}
void launch_mlp_step(float *, const float *, const float *, const float *, int64_t, float *,
                     float *, float *, float *, float *, float, float, float, cudaStream_t)
{
}
size_t mlp_grad_scratch_floats(int64_t) { return 1; }
int energy_work_size(int64_t) { return 1; }
int pair_step_slots(int64_t n, int64_t W) { return (int)(W / n) + 2; }
// blocks per SM, which differ from kernel to kernel
int pair_step_weak_blocks_per_sm(bool, WeakForm) { return 3; }
int pair_step_grp_weak_blocks_per_sm(bool, WeakForm) { return 3; }
int pair_step_sym_blocks_per_sm(bool, bool, bool seed, bool mixed) { return mixed ? 2 : (seed ? 3 : 4); }
int pair_step_grp_blocks_per_sm(bool, bool, bool, bool mixed) { return mixed ? 3 : 4; }
int pair_step_df64_blocks_per_sm(bool) { return 3; }
int pair_step_grp_df64_blocks_per_sm(bool) { return 1; }
int pair_step_grp_mixed_blocks_per_sm(bool, bool) { return 2; }
int pair_step_mixed_blocks_per_sm(bool) { return 2; }
int pair_step_fp64_blocks_per_sm(int, bool, bool) { return 4; }
int batched_blocks_per_sm(int, bool, bool, bool) { return 4; }

}  // namespace sakura
