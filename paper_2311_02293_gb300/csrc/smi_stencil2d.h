// smi_stencil2d.h -- single-launch 2D time steps (smi_stencil2d.cu).
#pragma once

#include <cuda.h>

#include "smi_internal.h"

namespace smi {

// Tensor maps of one batch's fields: pressure with the halo of a whole step,
// and the velocities with the halo of a whole reconstruction step.
struct Maps2 {
    CUtensorMap p, vz, vx;
};
// How a batch's steps are cut, chosen once a call by step2_tile from the
// points of a launch.
struct Step2 {
    bool many;             // enough tiles to fill the GPU several times
};
// Receivers' samples read by a forward step: p before the step is the
// pressure after step `it` (it < 0: none).
struct Gather2 {
    float *seis;
    const long long *off;  // [nshot] first sample of the shot
    int it;
};
// Boundary saving by a forward step: the velocities before the step become
// sample `sample` (negative: none); 16-bit storage scales by amax[sample]
// (device array [nsamp][nshot][6] of the largest magnitudes, zeroed before
// the first step), which the step before has filled; a step fills
// amax[next] (negative: none) with the velocities it writes.  amax null: a
// call that saves nothing.
struct Save2 {
    int sample, next;
    unsigned *amax;
};

// Adjoint source of the next reverse step (it: its step, negative: none), for
// the step kernel to add to the adjoint pressure it writes: residuals res at
// off[shot] + it nrec + r, and per shot the receivers whose stencils meet each
// cell of 32 columns (cell: [nshot][ncell + 1] positions in ids).
struct Inject2 {
    const float *res;
    const long long *off;
    const int *cell, *ids;
    int ncell, it;
};

bool stencil2d_supported(const Grid &g);
Step2 step2_tile(const Grid &g, int nshot);
// adjoint: maps of the adjoint fields (else of the source field).
bool make_maps2(Maps2 &m, const Grid &g, const Fields &f, int nshot, const Step2 &t, bool adjoint);

// One time step in one launch, from state c into state n (the same arrays'
// second set; memory variables included).  step = steps elapsed (the box).
// Forward: source stf (null: none), boundary saving, receiver samples.
void launch2_forward(const LaunchCtx &lc, const Step2 &t, const Maps2 &mc, const Grid &g, const Batch &b, Fields c,
                     Fields n, int step, const float *stf, float src_scale, const Bands &bd, Save2 save, Gather2 ga,
                     unsigned *err);
// Reverse: the adjoint step (mrev reverse steps elapsed) of (ac -> an)
// (roles & 1) and the reconstruction of the source field at step `it` (fc ->
// fn) with the imaging / gradient accumulation from ac's pressure (roles &
// 2).  restore: the band of step `it` from the store (every step stored).
void launch2_reverse(const LaunchCtx &lc, const Step2 &t, const Maps2 &mac, const Maps2 &mfc, const Grid &g,
                     const Batch &b, Fields ac, Fields an, int mrev, int roles, Fields fc, Fields fn, int it,
                     float *acc, int img_mode, const float *stf, float src_scale, const Bands &bd, bool restore,
                     Inject2 ij, unsigned *err);

}  // namespace smi
