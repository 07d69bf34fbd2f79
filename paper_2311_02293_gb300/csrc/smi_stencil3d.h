// smi_stencil3d.h -- TMA-streamed 3D stencil kernels (smi_stencil3d.cu).
#pragma once

#include <cuda.h>

#include "smi_internal.h"

namespace smi {

// Tensor maps of one batch's fields (haloed plane tiles and 32 x 16 core
// tiles), of the model arrays, and of the CPML slab arrays of the adjoint's
// operands (low and high slab; _p: on the p nodes, psiv, in the velocity
// kernel's geometry; _v: on the v nodes, psip, in the pressure kernel's).
struct Maps3 {
    CUtensorMap p_halo, p_core, vz_core, vx_core, vy_core, vz_halo, vx_halo, rho_v, K_core;
    CUtensorMap ezl_p, ezh_p, exl_p, exh_p, ezl_v, ezh_v, exl_v, exh_v;
};

// What the forward velocity kernel also does: receivers' samples of the
// pressure it reads, which is the pressure after step `it` (it < 0: none).
struct Gather3 {
    float *seis;
    const long long *off;
    int it;
};
// What the adjoint velocity kernel also does: the boundary of the source
// field v from the store's sample `it` (it < 0: none).
struct Restore3 {
    Bands bd;
    float *v[3];
    int it;
};
// What the forward pressure kernel also does: the velocities it reads become
// stored sample `sample` within bd's regions (16-bit storage scaled by the
// magnitudes in amax, which the velocity kernel has found), or, with find,
// their largest magnitudes per (shot, axis, side) go into amax (zeroed).
// sample < 0: none.
struct Save3 {
    Bands bd;
    unsigned *amax;
    int sample;
    bool find;
};

// One warp waits with the tile kernels' bounded-wait helper on an mbarrier
// that nothing completes, for `polls` polls, then sets bit 0 of err.
void launch_wait_check(const LaunchCtx &lc, unsigned *err, long long polls);
// The polls after which a tile kernel's wait gives up.
long long wait_polls_default();

// 4D tensor map (z, x, y, shot) over nshot padded fields starting at base,
// with a box of bz (z) x bx (x) x 1 x 1 and zero fill out of bounds; false if
// the encoder is missing or refuses the map.
bool make_tile_map(CUtensorMap *tm, const Grid &g, const float *base, int nshot, int bz, int bx);

// True when the tensor-map encoder was found.
bool tile_maps_available();

// True when the 3D kernels can run (3D, order 4 or 8, tensor-map encoder found).
bool stencil3d_supported(const Grid &g);

// Builds the maps for fields f of a batch of nshot shots (slabs: the CPML
// slab arrays too, in the tile kernels' layout); false on failure.
bool make_maps3(Maps3 &m, const Grid &g, const Fields &f, int nshot, bool slabs);

// mode 0: forward, 1: adjoint (step = reverse steps elapsed), 2: reconstruction.
// err: device word, bit 0 set if a bounded wait gave up; ctr: a zeroed device
// word of this launch (its work counter).  amax (forward, may be null): takes
// the largest magnitude per (shot, axis, side) of the band's velocities.
void launch3_v(const LaunchCtx &lc, const Maps3 &m, const Grid &g, const Batch &b, Fields f, int step, int mode,
               Gather3 ga, Restore3 rs, unsigned *amax, unsigned *err, unsigned *ctr);
// lpm: maps of the adjoint fields, whose pressure the reconstruction mode
// correlates with (mode 2 only).  stf null: no source.
void launch3_p(const LaunchCtx &lc, const Maps3 &m, const Maps3 *lpm, const Grid &g, const Batch &b, Fields f,
               int step, int mode, unsigned *err, float *acc, int img_mode, const float *stf, float src_scale, Save3 sv,
               unsigned *ctr);

}  // namespace smi
