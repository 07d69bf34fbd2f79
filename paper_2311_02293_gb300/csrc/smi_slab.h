// smi_slab.h -- CPML memory variables of the tile kernels: where the slabs of
// an axis lie in memory, and the recursion both directions share.
//
// Forward (Komatitsch & Martin): psi <- B psi + A D at the slab nodes, and
// D + psi takes the place of the derivative D.
// Adjoint: the transposed terms ask for D_a[q + A (q + m)] with m <- B (m + q)
// (q = lambda_p or lambda_v, m = phi or chi).  The kernels keep
// e = A (q + m) instead of m: then e <- B e + A q with the new q, the operand
// is q + e, and the neighbours read one value where m, A and q were needed.
// Both are the one recursion m <- B m + A x (slab_recur), with the
// coefficients of a node outside the slabs zero, so whole quads of four z
// nodes are updated without a test a node.
//
// Slab arrays of one shot (tile kernels; g.slab_n[a] floats each):
//   z: [y][x][js], quads of four z nodes aligned to 16 bytes: the low slab's
//      nodes 0 .. zlo-1 (zlo = nb rounded up to 4), then the nodes from zhi
//      (first node of the high slab rounded down to 4) to the row's end;
//   x: [y][js][z], rows of the field's pitch px, js = x < xlo or xlo + x - xhi;
//   y: [js][x][z], the same along y.
// An axis so short that one tile's stencil window could meet both slabs is
// stored whole (zlo = px, xlo = ne[1]: one slab).
#pragma once

#include "smi_internal.h"

namespace smi {

#ifdef __CUDACC__
// Offset of the z-slab quad that starts at node oz (a multiple of 4) inside
// its row of zp floats, or -1 when the quad holds no slab node.
__device__ __forceinline__ int zslab_quad(const Grid &g, int oz)
{
    if (oz < 0 || oz >= g.px) return -1;
    return oz < g.zlo ? oz : (oz >= g.zhi ? g.zlo + oz - g.zhi : -1);
}
// Index of node j inside the slab of axis a (1 or 2), or -1 outside.
__device__ __forceinline__ int slab_row(const Grid &g, int a, int j)
{
    const int lo = a == 1 ? g.xlo : g.nb, hi = a == 1 ? g.xhi : g.ne[a] - g.nb - 1;
    if (j < 0 || j >= g.ne[a]) return -1;
    return j < lo ? j : (j >= hi ? lo + j - hi : -1);
}
__device__ __forceinline__ float slab_recur(float B, float m, float A, float x) { return B * m + A * x; }
#endif

}  // namespace smi
