// sph_launch.h -- host-side launchers of the simulator kernels (internal).
#pragma once
#include <cuda_runtime.h>

#include "sph_common.cuh"

namespace sph {

// Launch with or without programmatic stream serialization.
template <typename... KArgs, typename... Args>
inline cudaError_t launch(void (*k)(KArgs...), int grid, int block, cudaStream_t st, bool pdl, Args... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = 0;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = pdl ? at : nullptr;
    cfg.numAttrs = pdl ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, k, args...);
}

void tile_dims(int code, int* tx, int* ty);
// Bytes of the per-tile staging records for the tile counts of every shape
// (n_tiles indexed by tile code 1..SPH_TILE_COUNT).
size_t stage_record_bytes(const int* n_tiles);
// pdl: launch with programmatic stream serialization (the kernels wait on
// their predecessor with griddepcontrol before reading its results).
// tan: the forward-mode tangent variants (tile codes 1..4 only).
// Phases: 0 density pass, 1 force pass, 2 body update.
// chained: this step directly follows a step of the same launch sequence
// (its density pass is the programmatic dependent of the previous step's
// body update), so that pass may stage the tile and sum the fluid part of
// Eq. 14 before its grid dependency: everything it reads there was written
// by the previous force pass, which completed before the body update passed
// its own dependency.
cudaError_t launch_phase(const SimDev& S, const EvalOut& E, int eval, int tile_code, int n_tiles, int phase,
                         cudaStream_t st, bool pdl, bool tan = false, bool chained = false);
cudaError_t launch_step(const SimDev& S, const EvalOut& E, int eval, int tile_code, int n_tiles, cudaStream_t st,
                        bool pdl, bool tan = false, bool chained = false);
// Phase 0 or 1 of a step on 4x4 tiles with four lanes per particle (sph_lanes.cu).
cudaError_t launch_lanes(const SimDev& S, int n_tiles, int phase, cudaStream_t st, bool pdl, int chained);
// Steps of small tanks in one launch (sph_resident.cu): whether a tank fits a
// cluster; the CTAs per tank for B tanks (0: not all at once), asked on the
// device before the first launch; n_steps steps under the run record already
// set, from the step that it stands at.
bool resident_fits(int n_f, int n_g, int G);
cudaError_t prepare_resident(int B, int& cluster);
cudaError_t launch_resident(const SimDev& S, int cluster, int n_steps, cudaStream_t st);
// State transfer: xv [N, 4] the hi parts of the particle state, lo [N, 4] its
// low parts (NULL: zero on binning, not read back on gathering).
cudaError_t launch_bin_flat(const SimDev& S, const float* xv, const float* lo, const int* part_tank, int n, int buf,
                            cudaStream_t st);
cudaError_t launch_set_body(const SimDev& S, const double* body, int buf, cudaStream_t st);
cudaError_t launch_get_state(const SimDev& S, float* xv, float* lo, double* body, int n_cells_total, int buf,
                             cudaStream_t st);
// Tangent state: with txv_out == NULL sets the tangent from txv_in / tb_in
// (NULL: zero); otherwise reads it into txv_out / tb_out.
cudaError_t launch_tangent_state(const SimDev& S, const float* txv_in, float* txv_out, const double* tb_in,
                                 double* tb_out, int n_cells_total, int buf, cudaStream_t st);
cudaError_t launch_set_run(RunDev* run, const RunDev& desc, cudaStream_t st);

// Recorded steps: their records lie step_bytes apart, their counts
// count_stride integers.  first: the SimDev of the first step, its arrays (of
// buffer buf0: the state binned at the body's position) in the first record.
// next_*: the state after the first step in the grid that the step left, in
// the first record (the state after step i, i records on).  Every `seg`th step
// starts a run: its state is already binned.
struct RecordDev {
    SimDev first;
    int buf0, seg;
    size_t step_bytes, count_stride;
    const float4 *next_pv, *next_lo;
    const int *next_pid, *next_count;
    int* flags;              // health flags of the tanks
    int flags_stride;        // integers between them
};
// The body records, re-binned states and density passes (4x4 tiles) of `steps` recorded steps.
cudaError_t launch_recorded(const RecordDev& R, const int* part_tank, int n_cells_total, int n_tiles, int steps,
                            cudaStream_t st);
// The health flags of `steps` reversed steps, and of the run that recorded them, to R.flags.
cudaError_t launch_record_flags(const RecordDev& R, const BodyDev* lane, int steps, cudaStream_t st);

// Reverse-mode step (sph_adjoint.cu) over a recorded step: S points at its
// records (launch_recorded), buf is the buffer of its state.  Adjoint arrays are indexed by particle index (the order of sph_get_state); body
// adjoints are (r_x, r_y, theta, rdot_x, rdot_y, thetadot).
struct AdjDev {
    const float4* in;        // [N] adjoint of (x, v) after the step
    float4* out;             // [N] adjoint of (x, v) before the step
    float* rhobar;           // [N] density adjoint (work)
    double* bbar;            // [B * 6] body adjoint: after the step on entry, before it on exit
    double* bbar_part;       // [B * 6] work: the integration part
    float* fbar;             // [B * 8] work: F_b, T_b and centre-of-mass adjoints of the step
    float* part;             // [2][max_tiles][12] work: per-tile body partials
    int max_tiles;
    const double* ybar;      // [B, n_samples, SPH_NY] sample adjoints (NULL: 0)
    long long ybar_stride;   // doubles between tanks
    double* ubar;            // [B, K, 3] input adjoints (NULL: not written)
    long long ubar_stride;
    int buf;                 // buffer of the state before the step
    int k;                   // step index within the call
    int row;                 // sample row of this step, -1: not sampled
};
int adjoint_tile_code();
// The body's part around a step: post finishes the step just reversed (its
// tile partials), pre begins step A.k (bbar, the samples and u of the step).
// pdl: the previous launch on st is a reverse step's too (the kernels stage
// from the records before they wait for it).
cudaError_t launch_adjoint_body(const SimDev& S, const AdjDev& A, int post, int pre, cudaStream_t st, bool pdl);
cudaError_t launch_adjoint_step(const SimDev& S, const AdjDev& A, int n_tiles, cudaStream_t st);
cudaError_t launch_set_step(RunDev* run, long long step, cudaStream_t st);

}  // namespace sph
