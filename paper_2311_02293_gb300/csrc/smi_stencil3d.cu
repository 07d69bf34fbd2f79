// smi_stencil3d.cu -- 3D staggered-grid stencil kernels for sm_103a.
//
// Two kernels advance one half of a leap-frog step each (Sec. 2.1 update
// equations): k3_v updates the three velocity components from p, k3_p
// updates p from the velocities.  Modes:
//   FWD  forward step on the computing box of the source, with the CPML
//        memory variables inline (Komatitsch & Martin) and the source;
//   ADJ  the exact discrete adjoint in "same solver" form on the box of the
//        receivers: the derivatives act on q + e, the operand of the
//        transposed CPML terms (smi_slab.h);
//   REC  source-field reconstruction backwards in time (Sec. 4.2) on the
//        physical domain, with the imaging / gradient accumulation fused
//        into the pressure kernel.
//
// Work decomposition: persistent CTAs (a fixed multiple of the SM count)
// draw the work items of the computing box (Sec. 4.1, evaluated on the device
// from the step counter; see Sched): 32 (z) x 16 (x) column tiles times
// chunks of y planes.  A CTA streams its chunk along y; a thread owns 4 consecutive
// z nodes of one x column.  Plane tiles arrive by TMA (cp.async.bulk.tensor;
// zeros outside the grid are the scheme's values there), issued two planes
// ahead as one group under one mbarrier:
//   velocity kernel, plane y: p of plane y+N with its z / x halo (ring of
//     N+2, since plane y's tile is needed N planes after it served the y
//     queue), the v tiles of plane y, rho of plane y+1;
//   pressure kernel, plane y: v_z and v_x with their halos, v_y of plane
//     y+N-1, p, kappa (and lambda_p) of plane y;
//   adjoint tiles that meet a z or x slab: e along z and x, halos included,
//     from the slab arrays (the TMA zero fill outside a slab is e = 0 there).
// y neighbours are kept in a register queue; z-derivatives read a 12-float
// window with three 128-bit shared loads, x-derivatives one 128-bit load a
// tap; multiplies and adds of the x and y derivatives run as packed pairs
// (f32x2, same rounding).
//
// What bounds them: the velocity kernel moves 32 B a point and the pressure
// kernel 24 (forward, adjoint) plus the halos that miss L2, so large boxes are
// bound by HBM (about 80 % of the copy rate) and small ones by the latency of
// a plane iteration.  Both ask for few instructions a point: box tests are
// folded into per-thread coefficients (a node outside the box has 2 dt = 0),
// ring positions are counted instead of divided, the last node's density is
// repeated in memory, one wait and one barrier serve a plane, and the planes
// without CPML terms run a body without them.  The loop body is not unrolled
// over planes: both bodies twice cost instruction-cache misses (four times:
// adjoint 0.88 of the rate).  The CPML terms ride on the tiles in flight
// instead of in kernels of their own over the slabs, which re-read the fields
// at half the bandwidth and took 26 % of a forward and 31 % of an adjoint step
// at 340^3 (50 % at 130^3).  A step of both kernels, GB300, with those kernels
// and now: 133 x 141 x 127, order 4, forward 77 -> 32 us; 200^3 extended,
// order 4, box on, 500 steps, forward 107 -> 77 us, adjoint 171 -> 98,
// reconstruction 67 -> 46; 340^3 extended, order 8, box on, first 600 steps,
// adjoint 378 -> 279, forward with 16-bit boundary saving 258 -> 179.
//
// Every mbarrier wait is bounded; a CTA that gives up issues no more copies,
// sets bit 0 of the error word, waits once more (bounded) for its copies in
// flight and returns.
#include <cuda.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "smi_band.h"
#include "smi_box.h"
#include "smi_internal.h"
#include "smi_pack.h"
#include "smi_pdl.h"
#include "smi_slab.h"
#include "smi_stencil3d.h"
#include "smi_tile3d.h"

namespace smi {
namespace s3 {

constexpr int CORE = TZ * TX;
constexpr int AHEAD = 2;             // planes by which plain loads of a later plane are prefetched into L2
// Plane groups in flight: two (42 - 53 KB of shared memory a CTA of the
// velocity kernel, four CTAs a SM); three were within 1 % either way.
constexpr int DEPTH = 2;

// Shared layouts in floats (every tile starts at a multiple of 128 bytes).
template <int N, int MODE> struct VLay {
    static constexpr int PR = TX + 2 * N - 1, PB = ZW * PR, P = rup32(PB), S = N + DEPTH;   // p: x0-N+1 .., z0-4 ..
    static constexpr int RB = 36 * (TX + 1), R = rup32(RB);                             // rho: x0 .. x0+TX, z0 .. z0+35
    static constexpr int EZ = ZW * TX, EXB = TZ * PR, EX = rup32(EXB);                  // e_z, e_x on p nodes
    static constexpr int oV = S * P, oR = oV + DEPTH * 3 * CORE, NR = DEPTH + 1, oE = oR + NR * R;
    static constexpr int SMEM = (oE + (MODE == ADJ ? DEPTH * (EZ + EX) : 0)) * 4;
};
template <int N, int MODE> struct PLay {
    static constexpr int Z = ZW * TX;                                  // v_z: z0-4 .., own x
    static constexpr int XR = TX + 2 * N - 1, XB = TZ * XR, X = rup32(XB);   // v_x: own z, x0-N ..
    static constexpr int oX = Z, oY = oX + X, oP = oY + CORE, oK = oP + CORE, oL = oK + CORE;
    static constexpr int oEZ = oL + (MODE == REC ? CORE : 0), oEX = oEZ + (MODE == ADJ ? Z : 0);
    static constexpr int G = oEX + (MODE == ADJ ? X : 0);              // one group
    static constexpr int SMEM = DEPTH * G * 4;
};

// CPML coefficients (B, A) of a tile's own nodes along z and x, zero at nodes
// outside the slabs, the grid or the box of this launch: a memory variable
// there stays what it is, zero.
struct alignas(16) Coefs {              // read as quads
    float zB[TZ], zA[TZ], xB[TX], xA[TX];
};
__device__ __forceinline__ void load_coefs(Coefs &c, const float *B0, const float *A0, const float *B1, const float *A1,
                                           const Item &it)
{
    for (int i = threadIdx.x; i < TZ + TX; i += NTHR) {
        if (i < TZ) {
            const int z = it.z0 + i;
            const bool in = in_range(z, it.lo[0], it.hi[0]);
            c.zB[i] = in ? B0[z] : 0.f;
            c.zA[i] = in ? A0[z] : 0.f;
        } else {
            const int x = it.x0 + i - TZ;
            const bool in = in_range(x, it.lo[1], it.hi[1]);
            c.xB[i - TZ] = in ? B1[x] : 0.f;
            c.xA[i - TZ] = in ? A1[x] : 0.f;
        }
    }
}

// A z slab (low, high) or x slab that the tile's stencil window reaches: its
// tensor map and the offset of its coordinates, or none.  The slabs of a
// short axis are one (smi_slab.h), so a window meets at most one.
struct SlabTile {
    const CUtensorMap *tm;
    int c;
};
__device__ __forceinline__ SlabTile z_slab_tile(const Grid &g, const CUtensorMap *lo, const CUtensorMap *hi, int z0)
{
    if (z0 - 4 < g.zlo) return {lo, z0 - 4};
    if (z0 + 36 > g.zhi) return {hi, z0 - 4 - g.zhi};
    return {nullptr, 0};
}
__device__ __forceinline__ SlabTile x_slab_tile(const Grid &g, const CUtensorMap *lo, const CUtensorMap *hi, int xs,
                                                int rows)
{
    if (xs < g.xlo) return {lo, xs};
    if (xs + rows > g.xhi) return {hi, xs - g.xhi};
    return {nullptr, 0};
}

// Per-thread position of an item.
struct Own {
    int oz, ox;
    bool act;                  // the quad's column lies in the grid and in the box along x
    int zq, xq;                // slab offsets of the own quad (-1: none)
};
__device__ __forceinline__ Own own_of(const Grid &g, const Item &it, int tzi, int txi)
{
    Own o;
    o.oz = it.z0 + 4 * tzi;
    o.ox = it.x0 + txi;
    o.act = o.oz < g.ne[0] && in_range(o.ox, it.lo[1], it.hi[1]);
    o.zq = o.act ? zslab_quad(g, o.oz) : -1;
    o.xq = o.act ? slab_row(g, 1, o.ox) : -1;
    return o;
}
// v - b D: the forward scheme rounds the product first (as it always has).
template <int MODE> __device__ __forceinline__ Q4 update(const Q4 &v, const Q4 &b, const Q4 &D)
{
    return MODE == FWD ? subq(v, mulq(b, D)) : fmaq(b, D, v);
}
// The forward scheme's z terms: which of the two products is rounded first
// decides the last bit.  A x enters the multiply-add unrounded, except on x
// lines whose group of four (from the low end of the shot's box) meets an x
// slab: a shot's bits are the same whichever shots it is launched with, and
// those of earlier kernels.
__device__ __forceinline__ void recur4z(bool xgroup, const float (&B)[4], const float (&A)[4], float (&m)[4], const Q4 &x)
{
    float v[4];
    split(x, v);
#pragma unroll
    for (int r = 0; r < 4; r++)
        m[r] = xgroup ? __fmaf_rn(B[r], m[r], __fmul_rn(A[r], v[r])) : __fmaf_rn(A[r], v[r], __fmul_rn(B[r], m[r]));
}
__device__ __forceinline__ bool x_group(const Grid &g, int x, int x0)
{
    const int first = x0 + ((x - x0) & ~3), hi = g.ne[1] - g.nb - 1;
    return first < g.nb || first + 3 >= hi;
}
// Maps of a launch, by the tile they bring.
struct VMaps {
    CUtensorMap p, rho, vz, vx, vy, ezl, ezh, exl, exh;
};
struct PMaps {
    CUtensorMap vz, vx, vy, p, K, lp, ezl, ezh, exl, exh;
};

// ===========================================================================
// Velocity kernel.  FWD / ADJ: v_a -= dt b_a D_a (p with its CPML term); REC:
// v_a += dt b_a D_a p on L_a+N-1..H_a-N, zero outside the previous box.
// MAG (FWD): the largest band magnitudes of the new velocities go into amax.
// Afterwards, by all CTAs: FWD the receivers' samples of p (step ga.it), ADJ
// the band of the source field from the store (rs.it).
template <int N, int MODE, bool MAG>
__global__ void __launch_bounds__(NTHR, SMI_MINB)
k3_v(const __grid_constant__ VMaps tm, Grid g, Batch b, Fields f, int step, int chunk, Gather3 ga, Restore3 rs,
     unsigned *amax, unsigned *err, unsigned *ctr)
{
    using La = VLay<N, MODE>;
    extern __shared__ __align__(128) float sm[];
    float *sv = sm + La::oV, *sr = sm + La::oR, *se = sm + La::oE;
    __shared__ __align__(8) uint64_t bar[DEPTH];
    __shared__ Coefs co;
    __shared__ unsigned smx[6];               // largest band magnitudes of the item (FWD with amax)
    __shared__ int next[2];                   // the CTA's next item, in turn
    const int tid = threadIdx.x, tzi = tid & 7, txi = tid >> 3;
    if (tid == 0) {
        for (int k = 0; k < DEPTH; k++) mbar_init(&bar[k], 1);
        mbar_fence_init();
    }
    if (tid < 6) smx[tid] = 0u;
    __syncthreads();
    Sched sd;
    sched_shot(g, b, MODE, step, 0, 0, chunk, sd);   // (the box tables are older than the loop)
    pdl_wait();
    pdl_trigger();
    unsigned phase = 0;                       // bit h: parity of the next completion of bar[h]
    bool ok = true;
    const float dt = g.dt;
    const int plane = g.px * g.ne[1];

    Item it;
    for (int w = blockIdx.x, par = 0; sched_item(g, b, MODE, step, w, chunk, sd, it); w = next[par], par ^= 1) {
        const int s = it.s, z0 = it.z0, x0 = it.x0, ya = it.ya, yb = it.yb;
        const Own me = own_of(g, it, tzi, txi);
        const int oz = me.oz, ox = me.ox;
        SlabTile ez{nullptr, 0}, ex{nullptr, 0};
        unsigned gbytes = (unsigned)(La::PB + 3 * CORE + La::RB) * 4u;
        if (MODE == ADJ) {
            ez = z_slab_tile(g, &tm.ezl, &tm.ezh, z0);
            ex = x_slab_tile(g, &tm.exl, &tm.exh, x0 - N + 1, La::PR);
            gbytes += (ez.tm ? La::EZ * 4u : 0u) + (ex.tm ? La::EXB * 4u : 0u);
        }
        // group of plane y: p(y+N), v(y), rho(y+1), e(y); ph = group slot
        auto issue = [&](int y, int ph, unsigned extra) {
            uint64_t *br = &bar[ph];
            mbar_expect(br, gbytes + extra);
            tma4(sm + ((y + N - ya) % La::S) * La::P, &tm.p, z0 - 4, x0 - N + 1, y + N, s, br);
            float *v = sv + ph * 3 * CORE;
            tma4(v, &tm.vz, z0, x0, y, s, br);
            tma4(v + CORE, &tm.vx, z0, x0, y, s, br);
            tma4(v + 2 * CORE, &tm.vy, z0, x0, y, s, br);
            tma4(sr + ((y + 1 - ya) % La::NR) * La::R, &tm.rho, z0, x0, y + 1, 0, br);
            if (MODE == ADJ) {
                float *e = se + ph * (La::EZ + La::EX);
                if (ez.tm) tma4(e, ez.tm, ez.c, x0, y, s, br);
                if (ex.tm) tma4(e + La::EZ, ex.tm, z0, ex.c, y, s, br);
            }
        };
        if (tid == 0 && ok) {
            issue(ya, 0, (unsigned)(N * La::PB + La::RB) * 4u);
            for (int l = 0; l < N; l++) tma4(sm + l * La::P, &tm.p, z0 - 4, x0 - N + 1, ya + l, s, &bar[0]);
            tma4(sr, &tm.rho, z0, x0, ya, 0, &bar[0]);
            for (int d = 1; d < DEPTH && ya + d <= yb; d++) issue(ya + d, d, 0u);
            next[par] = (int)(gridDim.x + atomicAdd(ctr, 1u));   // read after the item's last barrier
        }
        const long long sh = (long long)s * g.ntot;
        const unsigned col = (unsigned)(oz + g.px * ox);
        const bool grid_ok = oz < g.ne[0] && ox < g.ne[1];
        // y queue of own p: entry l = plane y-N+1+l; adjoint: p + e_y on the y-slab planes
        Q4 q[2 * N];
#pragma unroll
        for (int l = 0; l < 2 * N - 1; l++) {
            const int y = ya - N + 1 + l;
            q[l] = grid_ok && y >= 0 && y < g.ne[2] ? ldq(f.p + sh + (col + (unsigned)(y * plane))) : zeroq();
        }
        if (MODE == ADJ && me.act) {
#pragma unroll
            for (int l = 0; l < 2 * N - 1; l++) {
                const int js = slab_row(g, 2, ya - N + 1 + l);
                if (js >= 0) q[l] = addq(q[l], ldq(f.psiv[2] + s * g.slab_n[2] + (col + (unsigned)(js * plane))));
            }
        }
        // numerators of the buoyancy: 2 dt at the nodes a component updates, else 0 (adjoint and, along each
        // component's own range, reconstruction: signed so that the update is one multiply-add)
        Q4 mz, mx, mh;
        bool zc[4], hc[4];                    // REC: updated nodes outside the previous box along z and x
        bool clip = false;                    // REC: the tile has such nodes
        {
            const bool rx = MODE != REC || in_range(ox, g.L[1] + N - 1, g.H[1] - N);
            const float two = MODE == ADJ ? -2.0f * dt : 2.0f * dt;
            float a[4], c[4], h4[4];
#pragma unroll
            for (int r = 0; r < 4; r++) {
                const bool in = me.act && in_range(oz + r, it.lo[0], it.hi[0]);
                const bool rz = MODE != REC || in_range(oz + r, g.L[0] + N - 1, g.H[0] - N);
                a[r] = in && rz ? two : 0.f;
                c[r] = in && rx ? two : 0.f;
                h4[r] = in ? two : 0.f;
                const bool out = MODE == REC && in &&
                                 !(in_range(oz + r, it.plo[0], it.phi[0]) && in_range(ox, it.plo[1], it.phi[1]));
                hc[r] = out;
                zc[r] = out && rz;
                clip = clip || out;
            }
            mz = quad(a);
            mx = quad(c);
            mh = quad(h4);
        }
        const bool rxn = MODE == REC && in_range(ox, g.L[1] + N - 1, g.H[1] - N);
        if (MODE == REC) clip = __syncthreads_or(clip);
        if (MODE != REC) {
            load_coefs(co, g.cvb[0], g.cva[0], g.cvb[1], g.cva[1], it);
            __syncthreads();
        }
        // CPML planes of the item: every plane of a tile that meets a z or x slab, the y-slab planes of the others
        const bool zxb = MODE != REC && (z_slab_tile(g, &tm.p, &tm.p, z0).tm || x_slab_tile(g, &tm.p, &tm.p, x0 - N + 1, La::PR).tm);
        const bool xg = MODE == FWD && x_group(g, ox, it.lo[1]);
        // boundary bands (2N - 1 half nodes across each face): the quad's nodes per side of z, the side of x
        // that holds the column, the physical nodes; a plane's part is decided per plane
        unsigned bz0 = 0u, bz1 = 0u, bph = 0u;
        int bxs = -1;
        bool bzt = false, bxt = false;         // the tile meets a z band, an x band
        if (MAG) {
            constexpr unsigned W = 2 * N - 2;
            const bool px = me.act && in_range(ox, g.L[1], g.H[1]);
#pragma unroll
            for (int r = 0; r < 4; r++) {
                bz0 |= px && (unsigned)(oz + r - g.L[0] + N) <= W ? 1u << r : 0u;
                bz1 |= px && (unsigned)(oz + r - g.H[0] + N - 1) <= W ? 1u << r : 0u;
                bph |= me.act && in_range(oz + r, g.L[0], g.H[0]) ? 1u << r : 0u;
            }
            bxs = (unsigned)(ox - g.L[1] + N) <= W ? 0 : ((unsigned)(ox - g.H[1] + N - 1) <= W ? 1 : -1);
            bzt = (z0 <= g.L[0] + N - 2 && z0 + TZ - 1 >= g.L[0] - N) || (z0 <= g.H[0] + N - 1 && z0 + TZ - 1 >= g.H[0] - N + 1);
            bxt = (x0 <= g.L[1] + N - 2 && x0 + TX - 1 >= g.L[1] - N) || (x0 <= g.H[1] + N - 1 && x0 + TX - 1 >= g.H[1] - N + 1);
        }
        auto note = [&](int k, const Q4 &v, unsigned mask) {      // uniform call
            const unsigned u = warp_max(v, mask);
            if ((tid & 31) == 0 && u) atomicMax(&smx[k], u);
        };
        const bool lastz = oz + 4 >= g.px;
        const int rxrow = ox + 1 < g.ne[1] ? txi + 1 : txi;        // the last node's neighbour is itself
        float *const mzp = f.psip[0] + (s * g.slab_n[0] + me.zq + (long long)g.zp * ox);
        float *const mxp = f.psip[1] + (s * g.slab_n[1] + oz + (long long)g.px * me.xq);
        const unsigned zpl = (unsigned)(g.zp * g.ne[1]), xpl = (unsigned)(g.px * g.xrows);
        int h = 0, kp = 0, kq = N % La::S, kr = 0;   // group, ring slots of p(y), p(y+N), rho(y)

        // one plane; BAND: with the CPML terms (REC: with nodes outside the previous box)
        auto body = [&](auto kc, auto bc, int y) {
            constexpr int K = decltype(kc)::value;
            constexpr bool BAND = decltype(bc)::value;
            const int ys = BAND && MODE != REC ? slab_row(g, 2, y) : -1;
            const int ye = BAND && MODE == ADJ ? slab_row(g, 2, y + N) : -1;
            float ym[4], mzv[4], mxv[4];
            Q4 yp;
            if (BAND && MODE != REC) {
                if (ys >= 0 && me.act) put(ym, ldg4(f.psip[2] + s * g.slab_n[2] + (col + (unsigned)(ys * plane))));
                if (ye >= 0 && me.act) yp = ldq(f.psiv[2] + s * g.slab_n[2] + (col + (unsigned)(ye * plane)));
                if (me.xq >= 0) put(mxv, ldg4(mxp + (unsigned)y * xpl));
                if (me.zq >= 0) put(mzv, ldg4(mzp + (unsigned)y * zpl));
                if (y + AHEAD <= yb) {
                    if (me.xq >= 0) prefetch_l2(mxp + (unsigned)(y + AHEAD) * xpl);
                    if (me.zq >= 0) prefetch_l2(mzp + (unsigned)(y + AHEAD) * zpl);
                }
            }
            ok = ok && mbar_wait(&bar[h], (phase >> h) & 1u);
            phase ^= 1u << h;
            const float *pt = sm + kp * La::P + (txi + N - 1) * ZW + 4 * tzi;      // window of the own quad
            const int kr1 = kr == La::NR - 1 ? 0 : kr + 1;
            const float *rt = sr + kr * La::R + 4 * tzi;
            const float *cs = sv + h * 3 * CORE + txi * TZ + 4 * tzi;
            Q4 &qn = q[(2 * N - 1 + K) % (2 * N)];
            qn = ldq(sm + kq * La::P + (txi + N - 1) * ZW + 4 * tzi + 4);
            if (BAND && ye >= 0 && me.act) qn = addq(qn, yp);
            const Q4 r0 = ldq(rt + txi * 36);
            const unsigned o = col + (unsigned)(y * plane);
            const bool ky = !(BAND && MODE == REC) || in_range(y, it.plo[2], it.phi[2]);

            // ---- y component ----
            if (MODE != REC || in_range(y, g.L[2] + N - 1, g.H[2] - N)) {
                Q4 D = zeroq();
#pragma unroll
                for (int l = 1; l <= N; l++) D = tap(D, g.c[2][l - 1], q[(N - 1 + l + K) % (2 * N)], q[(N - l + K) % (2 * N)]);
                const Q4 r1 = ldq((y + 1 < g.ne[2] ? sr + kr1 * La::R : sr + kr * La::R) + txi * 36 + 4 * tzi);
                const Q4 bb = buoyq(mh, r0, r1);
                Q4 v = ldq(cs + 2 * CORE);
                if (BAND && MODE != REC && ys >= 0 && me.act) {
                    float B[4], A[4], m[4];
                    split(mh, m);
#pragma unroll
                    for (int r = 0; r < 4; r++) {
                        B[r] = g.cvb[2][y];
                        A[r] = m[r] != 0.f ? g.cva[2][y] : 0.f;
                    }
                    if (MODE == FWD) {
                        recur4(B, A, ym, D);
                        D = addq(D, quad(ym));
                    }
                    v = update<MODE>(v, bb, D);
                    if (MODE == ADJ) recur4(B, A, ym, v);
                    stg4(f.psip[2] + s * g.slab_n[2] + (col + (unsigned)(ys * plane)), ym);
                } else {
                    v = update<MODE>(v, bb, D);
                }
                if (BAND && MODE == REC) {
                    float m[4];
                    bool cl[4];
                    split(mh, m);
#pragma unroll
                    for (int r = 0; r < 4; r++) cl[r] = hc[r] || (!ky && m[r] != 0.f);
                    v = clear_if(v, cl);
                }
                if (me.act) stq(f.v[2] + sh + o, v);
                if (BAND && MAG) {
                    const unsigned in = in_range(ox, g.L[1], g.H[1]) ? bph : 0u;
                    if ((unsigned)(y - g.L[2] + N) <= 2 * N - 2) note(4, v, in);
                    if ((unsigned)(y - g.H[2] + N - 1) <= 2 * N - 2) note(5, v, in);
                }
            }
            float W[12];
            window(W, pt);
            // ---- x component ----
            {
                Q4 D = zeroq();
                const float *er = se + h * (La::EZ + La::EX) + La::EZ + (txi + N - 1) * TZ + 4 * tzi;
#pragma unroll
                for (int l = 1; l <= N; l++) {
                    Q4 a = ldq(pt + 4 + l * ZW);
                    Q4 c = l == 1 ? quad({W[4], W[5], W[6], W[7]}) : ldq(pt + 4 - (l - 1) * ZW);
                    if (BAND && MODE == ADJ && ex.tm) {
                        a = addq(a, ldq(er + l * TZ));
                        c = addq(c, ldq(er - (l - 1) * TZ));
                    }
                    D = tap(D, g.c[1][l - 1], a, c);
                }
                const Q4 bb = buoyq(mx, r0, ldq(rt + rxrow * 36));
                Q4 v = update<MODE>(ldq(cs + CORE), bb, D);
                if (BAND && MODE != REC && me.xq >= 0) {
                    recur1(co.xB[txi], co.xA[txi], mxv, MODE == FWD ? D : v);
                    if (MODE == FWD) v = sub_prod(v, bb, mxv);
                    stg4(mxp + (unsigned)y * xpl, mxv);
                }
                if (BAND && MODE == REC && rxn) {
                    float m[4];
                    bool cl[4];
                    split(mh, m);
#pragma unroll
                    for (int r = 0; r < 4; r++) cl[r] = hc[r] || (!ky && m[r] != 0.f);
                    v = clear_if(v, cl);
                }
                if (me.act) stq(f.v[1] + sh + o, v);
                if (BAND && MAG && bxt && in_range(y, g.L[2], g.H[2])) {
                    note(2, v, bxs == 0 ? bph : 0u);
                    note(3, v, bxs == 1 ? bph : 0u);
                }
            }
            // ---- z component ----
            {
                if (BAND && MODE == ADJ && ez.tm) {
                    float E[12];
                    window(E, se + h * (La::EZ + La::EX) + txi * ZW + 4 * tzi);
#pragma unroll
                    for (int i = 0; i < 12; i++) W[i] += E[i];
                }
                const Q4 D = dz4<N, true>(g, W);
                float ra[4];
                split(r0, ra);
                const Q4 r1 = quad({ra[1], ra[2], ra[3], lastz ? ra[3] : rt[txi * 36 + 4]});
                const Q4 bb = buoyq(mz, r0, r1);
                Q4 v = update<MODE>(ldq(cs), bb, D);
                if (BAND && MODE != REC && me.zq >= 0) {
                    float B[4], A[4];
                    put(B, lds4(co.zB + 4 * tzi));
                    put(A, lds4(co.zA + 4 * tzi));
                    if (MODE == FWD) recur4z(xg, B, A, mzv, D);
                    else recur4(B, A, mzv, v);
                    if (MODE == FWD) v = sub_prod(v, bb, mzv);
                    stg4(mzp + (unsigned)y * zpl, mzv);
                }
                if (BAND && MODE == REC) {
                    float m[4];
                    bool cl[4];
                    split(mz, m);
#pragma unroll
                    for (int r = 0; r < 4; r++) cl[r] = zc[r] || (!ky && m[r] != 0.f);
                    v = clear_if(v, cl);
                }
                if (me.act) stq(f.v[0] + sh + o, v);
                if (BAND && MAG && bzt && in_range(y, g.L[2], g.H[2])) {
                    note(0, v, bz0);
                    note(1, v, bz1);
                }
            }
            kp = kp + 1 == La::S ? 0 : kp + 1;
            kq = kq + 1 == La::S ? 0 : kq + 1;
            kr = kr1;
            __syncthreads();                  // every read of plane y's tiles is done
            if (tid == 0 && ok && y + DEPTH <= yb) issue(y + DEPTH, h, 0u);
            h = h + 1 == DEPTH ? 0 : h + 1;
        };
        auto one = [&](auto kc, int y) {
            const bool band = MODE == REC ? clip || !in_range(y, it.plo[2], it.phi[2])
                                          : zxb || yslab(g, y) || (MODE == ADJ && yslab(g, y + N)) ||
                                                (MAG &&
                                                 (bzt || bxt || (unsigned)(y - g.L[2] + N) <= 2 * N - 2 ||
                                                  (unsigned)(y - g.H[2] + N - 1) <= 2 * N - 2));
            if (band) body(kc, std::true_type{}, y);
            else body(kc, std::false_type{}, y);
        };
        constexpr int G = (2 * N) % SMI_YUNROLL == 0 ? SMI_YUNROLL : 2 * N;
        for (int y = ya; y <= yb; y += G) {
            unroll_planes<G>(one, y, yb);
            rotate_queue<G>(q);
        }
        if (__syncthreads_or(!ok)) break;
        if (MAG && tid < 6 && smx[tid]) {         // (the next item notes nothing before its barrier)
            atomicMax(amax + s * 6 + tid, smx[tid]);
            smx[tid] = 0u;
        }
    }
    if (__syncthreads_or(!ok)) {
        if (tid == 0) atomicOr(err, 1u);
        for (int k = 0; k < DEPTH; k++) mbar_wait(&bar[k], (phase >> k) & 1u);
        return;
    }
    if (MODE == FWD && ga.it >= 0) gather_tail(g, b, f.p, ga);
    if (MODE == ADJ && rs.it >= 0) restore_tail(g, b.nshot, rs);
}

// ===========================================================================
// Pressure kernel.  FWD / ADJ: p -= dt kappa sum_a D_a (v_a with its CPML
// term), FWD with the source; REC: acc += lp * (div v | p), p += dt kappa div v
// - source, zero outside the previous box, on the physical domain.
// Afterwards FWD, by all CTAs: the next stored boundary (or its largest
// magnitudes), from the velocities this kernel only reads.
template <int N, int MODE>
__global__ void __launch_bounds__(NTHR, SMI_MINB)
k3_p(const __grid_constant__ PMaps tm, Grid g, Batch b, Fields f, int step, int chunk, unsigned *err, float *acc, int img_mode,
     const float *stf, float src_scale, Save3 sv, unsigned *ctr)
{
    using La = PLay<N, MODE>;
    extern __shared__ __align__(128) float sm[];
    __shared__ __align__(8) uint64_t bar[DEPTH];
    __shared__ Coefs co;
    __shared__ int next[2];                   // the CTA's next item, in turn
    const int tid = threadIdx.x, tzi = tid & 7, txi = tid >> 3;
    if (tid == 0) {
        for (int k = 0; k < DEPTH; k++) mbar_init(&bar[k], 1);
        mbar_fence_init();
    }
    __syncthreads();
    Sched sd;
    sched_shot(g, b, MODE, step, 0, 0, chunk, sd);   // (the box tables are older than the loop)
    pdl_wait();
    pdl_trigger();
    unsigned phase = 0;
    bool ok = true;
    const float dt = g.dt;
    const int plane = g.px * g.ne[1];

    Item it;
    for (int w = blockIdx.x, par = 0; sched_item(g, b, MODE, step, w, chunk, sd, it); w = next[par], par ^= 1) {
        const int s = it.s, z0 = it.z0, x0 = it.x0, ya = it.ya, yb = it.yb;
        const Own me = own_of(g, it, tzi, txi);
        const int oz = me.oz, ox = me.ox;
        SlabTile ez{nullptr, 0}, ex{nullptr, 0};
        unsigned gbytes = (unsigned)(La::Z + La::XB + (MODE == REC ? 4 : 3) * CORE) * 4u;
        if (MODE == ADJ) {
            ez = z_slab_tile(g, &tm.ezl, &tm.ezh, z0);
            ex = x_slab_tile(g, &tm.exl, &tm.exh, x0 - N, La::XR);
            gbytes += (ez.tm ? La::Z * 4u : 0u) + (ex.tm ? La::XB * 4u : 0u);
        }
        auto issue = [&](int y, int ph) {
            uint64_t *br = &bar[ph];
            float *t = sm + ph * La::G;
            mbar_expect(br, gbytes);
            tma4(t, &tm.vz, z0 - 4, x0, y, s, br);
            tma4(t + La::oX, &tm.vx, z0, x0 - N, y, s, br);
            tma4(t + La::oY, &tm.vy, z0, x0, y + N - 1, s, br);
            tma4(t + La::oP, &tm.p, z0, x0, y, s, br);
            tma4(t + La::oK, &tm.K, z0, x0, y, 0, br);
            if (MODE == REC) tma4(t + La::oL, &tm.lp, z0, x0, y, s, br);
            if (MODE == ADJ) {
                if (ez.tm) tma4(t + La::oEZ, ez.tm, ez.c, x0, y, s, br);
                if (ex.tm) tma4(t + La::oEX, ex.tm, z0, ex.c, y, s, br);
            }
        };
        if (tid == 0 && ok) {
            issue(ya, 0);
            for (int d = 1; d < DEPTH && ya + d <= yb; d++) issue(ya + d, d);
            next[par] = (int)(gridDim.x + atomicAdd(ctr, 1u));
        }
        const long long sh = (long long)s * g.ntot;
        const unsigned col = (unsigned)(oz + g.px * ox);
        const bool grid_ok = oz < g.ne[0] && ox < g.ne[1];
        // y queue of own v_y: entry l = plane y-N+l; adjoint: v_y + e_y on the y-slab planes
        Q4 q[2 * N];
#pragma unroll
        for (int l = 0; l < 2 * N - 1; l++) {
            const int y = ya - N + l;
            q[l] = grid_ok && y >= 0 && y < g.ne[2] ? ldq(f.v[2] + sh + (col + (unsigned)(y * plane))) : zeroq();
        }
        if (MODE == ADJ && me.act) {
#pragma unroll
            for (int l = 0; l < 2 * N - 1; l++) {
                const int js = slab_row(g, 2, ya - N + l);
                if (js >= 0) q[l] = addq(q[l], ldq(f.psip[2] + s * g.slab_n[2] + (col + (unsigned)(js * plane))));
            }
        }
        Q4 md;                                // dt at the nodes of the update region, else 0 (adjoint: -dt)
        bool in[4], out[4];                   // REC: updated nodes, and those outside the previous box along z and x
        bool clip = false;
        {
            float a[4];
#pragma unroll
            for (int r = 0; r < 4; r++) {
                in[r] = me.act && in_range(oz + r, it.lo[0], it.hi[0]);
                a[r] = in[r] ? (MODE == ADJ ? -dt : dt) : 0.f;
                out[r] = MODE == REC && in[r] &&
                         !(in_range(oz + r, it.plo[0], it.phi[0]) && in_range(ox, it.plo[1], it.phi[1]));
                clip = clip || out[r];
            }
            md = quad(a);
        }
        // whether the source stencil reaches this item's tile column and y range
        bool src_col = false;
        float amp = 0.f;
        if (MODE != ADJ && stf) {
            const Stencil &st = b.src[s];
            src_col = st.first[0] <= z0 + TZ - 1 && st.first[0] + st.cnt[0] - 1 >= z0 && st.first[1] <= x0 + TX - 1 &&
                      st.first[1] + st.cnt[1] - 1 >= x0 && st.first[2] <= yb && st.first[2] + st.cnt[2] - 1 >= ya;
            amp = (MODE == REC ? -src_scale : src_scale) * stf[step];
        }
        if (MODE == REC) clip = __syncthreads_or(clip);
        if (MODE != REC) {
            load_coefs(co, g.cpb[0], g.cpa[0], g.cpb[1], g.cpa[1], it);
            __syncthreads();
        }
        const bool zxb = MODE != REC && (z_slab_tile(g, &tm.p, &tm.p, z0).tm || x_slab_tile(g, &tm.p, &tm.p, x0 - N, La::XR).tm);
        const bool xg = MODE == FWD && x_group(g, ox, it.lo[1]);
        float *const mzp = f.psiv[0] + (s * g.slab_n[0] + me.zq + (long long)g.zp * ox);
        float *const mxp = f.psiv[1] + (s * g.slab_n[1] + oz + (long long)g.px * me.xq);
        const unsigned zpl = (unsigned)(g.zp * g.ne[1]), xpl = (unsigned)(g.px * g.xrows);
        int h = 0;                            // group slot of plane y

        // one plane; BAND: with the CPML terms (REC: with nodes outside the previous box)
        auto body = [&](auto kc, auto bc, int y) {
            constexpr int K = decltype(kc)::value;
            constexpr bool BAND = decltype(bc)::value;
            const unsigned o = col + (unsigned)(y * plane);
            Q4 accv = zeroq();
            if (MODE == REC && me.act) {
                if (y + AHEAD <= yb) prefetch_l2(acc + sh + (o + (unsigned)(AHEAD * plane)));
                accv = ldq(acc + sh + o);
            }
            const int ys = BAND && MODE != REC ? slab_row(g, 2, y) : -1;
            const int ye = BAND && MODE == ADJ ? slab_row(g, 2, y + N - 1) : -1;
            float ym[4], mzv[4], mxv[4];
            Q4 yc;
            if (BAND && MODE != REC) {
                if (ys >= 0 && me.act) put(ym, ldg4(f.psiv[2] + s * g.slab_n[2] + (col + (unsigned)(ys * plane))));
                if (ye >= 0 && me.act) yc = ldq(f.psip[2] + s * g.slab_n[2] + (col + (unsigned)(ye * plane)));
                if (me.xq >= 0) put(mxv, ldg4(mxp + (unsigned)y * xpl));
                if (me.zq >= 0) put(mzv, ldg4(mzp + (unsigned)y * zpl));
                if (y + AHEAD <= yb) {
                    if (me.xq >= 0) prefetch_l2(mxp + (unsigned)(y + AHEAD) * xpl);
                    if (me.zq >= 0) prefetch_l2(mzp + (unsigned)(y + AHEAD) * zpl);
                }
            }
            ok = ok && mbar_wait(&bar[h], (phase >> h) & 1u);
            phase ^= 1u << h;
            const float *t = sm + h * La::G, *own = t + txi * TZ + 4 * tzi;
            Q4 &qn = q[(2 * N - 1 + K) % (2 * N)];
            qn = ldq(own + La::oY);
            if (BAND && ye >= 0 && me.act) qn = addq(qn, yc);
            // ---- y ----
            Q4 Dy = zeroq();
#pragma unroll
            for (int l = 1; l <= N; l++) Dy = tap(Dy, g.c[2][l - 1], q[(N + l - 1 + K) % (2 * N)], q[(N - l + K) % (2 * N)]);
            float By = 0.f, Ay[4] = {0.f, 0.f, 0.f, 0.f};          // y memory variable
            if (BAND && MODE != REC && ys >= 0 && me.act) {
                By = g.cpb[2][y];
#pragma unroll
                for (int r = 0; r < 4; r++) Ay[r] = in[r] ? g.cpa[2][y] : 0.f;
                if (MODE == FWD) {
                    const float B4[4] = {By, By, By, By};
                    recur4(B4, Ay, ym, Dy);
                    Dy = addq(Dy, quad(ym));
                }
            }
            // ---- x ----
            Q4 Dx = zeroq();
            {
                const float *xr = t + La::oX + (txi + N) * TZ + 4 * tzi, *er = t + La::oEX + (txi + N) * TZ + 4 * tzi;
#pragma unroll
                for (int l = 1; l <= N; l++) {
                    Q4 a = ldq(xr + (l - 1) * TZ), c = ldq(xr - l * TZ);
                    if (BAND && MODE == ADJ && ex.tm) {
                        a = addq(a, ldq(er + (l - 1) * TZ));
                        c = addq(c, ldq(er - l * TZ));
                    }
                    Dx = tap(Dx, g.c[1][l - 1], a, c);
                }
            }
            // ---- z ----
            Q4 div;
            {
                float W[12];
                window(W, t + txi * ZW + 4 * tzi);
                if (BAND && MODE == ADJ && ez.tm) {
                    float E[12];
                    window(E, t + La::oEZ + txi * ZW + 4 * tzi);
#pragma unroll
                    for (int i = 0; i < 12; i++) W[i] += E[i];
                }
                div = dz4<N, false>(g, W);
            }
            if (BAND && MODE == FWD) {
                if (me.zq >= 0) {
                    float B[4], A[4];
                    put(B, lds4(co.zB + 4 * tzi));
                    put(A, lds4(co.zA + 4 * tzi));
                    recur4z(xg, B, A, mzv, div);
                    stg4(mzp + (unsigned)y * zpl, mzv);
                }
                if (me.xq >= 0) {
                    recur1(co.xB[txi], co.xA[txi], mxv, Dx);
                    stg4(mxp + (unsigned)y * xpl, mxv);
                }
            }
            div = addq(addq(div, Dx), Dy);
            const Q4 pv = ldq(own + La::oP), dK = mulq(md, ldq(own + La::oK));
            Q4 np = update<MODE>(pv, dK, div);
            if (BAND && MODE == FWD && (me.zq >= 0 || me.xq >= 0)) {
                // z and x memory variables: their own product, after the plain derivatives'
                float m[4];
#pragma unroll
                for (int r = 0; r < 4; r++) m[r] = (me.zq >= 0 ? mzv[r] : 0.f) + (me.xq >= 0 ? mxv[r] : 0.f);
                np = sub_prod(np, dK, m);
            }
            if (MODE != ADJ && src_col) {
                const Stencil &st = b.src[s];
                const int t1 = ox - st.first[1], t2 = y - st.first[2];
                if (t1 >= 0 && t1 < st.cnt[1] && t2 >= 0 && t2 < st.cnt[2]) {
                    float x[4];
                    split(np, x);
#pragma unroll
                    for (int r = 0; r < 4; r++) {
                        const int t0 = oz + r - st.first[0];
                        if (t0 >= 0 && t0 < st.cnt[0] && (MODE == FWD || in[r]))
                            x[r] += amp * (st.w[0][t0] * st.w[1][t1] * st.w[2][t2]);
                    }
                    np = quad(x);
                }
            }
            if (MODE == REC) {
                // (div v reaches past the box, p does not; outside the physical domain p gathers what nobody reads)
                bool off[4];
#pragma unroll
                for (int r = 0; r < 4; r++) off[r] = !in[r];
                if (me.act) stq(acc + sh + o, fmaq(ldq(own + La::oL), img_mode == 0 ? clear_if(div, off) : pv, accv));
                if (img_mode == 2 && me.act) {                // illumination
                    float *ill = acc + (long long)b.nshot * g.ntot + sh + o;
                    stq(ill, fmaq(pv, pv, ldq(ill)));
                }
                if (BAND) {
                    const bool ky = in_range(y, it.plo[2], it.phi[2]);
                    bool cl[4];
#pragma unroll
                    for (int r = 0; r < 4; r++) cl[r] = out[r] || (!ky && in[r]);
                    np = clear_if(np, cl);
                }
            }
            if (BAND && MODE == ADJ) {
                if (me.zq >= 0) {
                    float Bz[4], Az[4];
                    put(Bz, lds4(co.zB + 4 * tzi));
                    put(Az, lds4(co.zA + 4 * tzi));
                    recur4(Bz, Az, mzv, np);
                    stg4(mzp + (unsigned)y * zpl, mzv);
                }
                if (me.xq >= 0) {
                    recur1(co.xB[txi], co.xA[txi], mxv, np);
                    stg4(mxp + (unsigned)y * xpl, mxv);
                }
                if (ys >= 0 && me.act) {
                    const float B4[4] = {By, By, By, By};
                    recur4(B4, Ay, ym, np);
                }
            }
            if (BAND && MODE != REC && ys >= 0 && me.act)
                stg4(f.psiv[2] + s * g.slab_n[2] + (col + (unsigned)(ys * plane)), ym);
            if (me.act) stq(f.p + sh + o, np);
            __syncthreads();
            if (tid == 0 && ok && y + DEPTH <= yb) issue(y + DEPTH, h);
            h = h + 1 == DEPTH ? 0 : h + 1;
        };
        auto one = [&](auto kc, int y) {
            const bool band = MODE == REC ? clip || !in_range(y, it.plo[2], it.phi[2])
                                          : zxb || yslab(g, y) || (MODE == ADJ && yslab(g, y + N - 1));
            if (band) body(kc, std::true_type{}, y);
            else body(kc, std::false_type{}, y);
        };
        constexpr int G = (2 * N) % SMI_YUNROLL == 0 ? SMI_YUNROLL : 2 * N;
        for (int y = ya; y <= yb; y += G) {
            unroll_planes<G>(one, y, yb);
            rotate_queue<G>(q);
        }
        if (__syncthreads_or(!ok)) break;
    }
    if (__syncthreads_or(!ok)) {
        if (tid == 0) atomicOr(err, 1u);
        for (int k = 0; k < DEPTH; k++) mbar_wait(&bar[k], (phase >> k) & 1u);
        return;
    }
    if (MODE == FWD && sv.sample >= 0) save_tail(g, b.nshot, f, sv);
}

// Give-up path of the bounded waits: one warp waits, with the tile kernels'
// own wait helper, on an mbarrier that nothing completes; when the polls run
// out it records the give-up in err like a tile kernel does, and returns.
__global__ void k_wait_check(unsigned *err, long long polls)
{
    __shared__ __align__(8) uint64_t bar;
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        mbar_fence_init();
    }
    __syncthreads();
    const bool ok = mbar_wait(&bar, 0u, polls);
    if (!ok && threadIdx.x == 0) atomicOr(err, 1u);
}

}  // namespace s3


// ---------------------------------------------------------------------------
// Host side: tensor maps and launches.

namespace {

using EncodeFn = CUresult (*)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                              const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                              CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeFn encoder()
{
    // initialised once, by the first thread; others wait (the server's slots start together)
    static const EncodeFn fn = []() -> EncodeFn {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            return reinterpret_cast<EncodeFn>(p);
        cudaGetLastError();
        return nullptr;
    }();
    return fn;
}

// 4D map (z, x, y, shot) over a padded field array with a box of bz x bx x 1 x 1.
bool make_map(CUtensorMap *tm, const Grid &g, const float *base, int nshot, int bz, int bx)
{
    EncodeFn fn = encoder();
    if (!fn) return false;
    cuuint64_t dims[4] = {(cuuint64_t)g.ne[0], (cuuint64_t)g.ne[1], (cuuint64_t)g.ne[2], (cuuint64_t)nshot};
    cuuint64_t strides[3] = {(cuuint64_t)g.px * 4, (cuuint64_t)g.px * g.ne[1] * 4,
                             (cuuint64_t)g.px * g.ne[1] * g.ne[2] * 4};
    cuuint32_t box[4] = {(cuuint32_t)bz, (cuuint32_t)bx, 1, 1};
    cuuint32_t es[4] = {1, 1, 1, 1};
    CUresult r = fn(tm, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, const_cast<float *>(base), dims, strides, box, es,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS;
}

// 4D map over a slab array (n0, n1, n2, shot) with strides in floats.
bool make_slab_map(CUtensorMap *tm, const float *base, int n0, int n1, int n2, int nshot, long long s1, long long s2,
                   long long sshot, int b0, int b1)
{
    EncodeFn fn = encoder();
    if (!fn) return false;
    cuuint64_t dims[4] = {(cuuint64_t)n0, (cuuint64_t)n1, (cuuint64_t)n2, (cuuint64_t)nshot};
    cuuint64_t strides[3] = {(cuuint64_t)s1 * 4, (cuuint64_t)s2 * 4, (cuuint64_t)sshot * 4};
    cuuint32_t box[4] = {(cuuint32_t)b0, (cuuint32_t)b1, 1, 1};
    cuuint32_t es[4] = {1, 1, 1, 1};
    return fn(tm, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, const_cast<float *>(base), dims, strides, box, es,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <class K> int grid_for(K kernel, int smem)
{
    cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
    int per = 0, dev = 0, sms = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kernel, s3::NTHR, smem);
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return std::max(1, per) * std::max(1, sms);
}

// Planes a chunk of a launch over `cols` tile columns (all shots) of ylen
// planes.  Large launches: 8 planes (more when that makes over eight items a
// CTA), so that the sweep stays local (see Sched).  Launches of one to four
// 8-plane items a CTA: four items a CTA, of 5 planes or more -- items differ in
// cost (CPML planes, cut tiles), and the CTAs that draw cheap ones take over
// (12 planes, or 8 planes in a wave and a part, before: 160^3 migration order 4
// 115.9 -> 107.5 ms, 131 x 243 x 205 162.2 -> 157.9, 93 x 101 x 87 forward 13.18 ->
// 12.72; three items a CTA 108.7, 158.4, 12.92).  Smaller ones, whose items
// run at once: the chunk between 8 and 24 planes that finishes first when an
// item costs its planes plus a start of about 7, and an SM runs three items
// as fast as one (measured on 133 x 141 x 127 points, order 4, a step: 22
// planes 44 us, 15 planes 33, 12 planes 37, 8 planes 34).
int pick_chunk(long long cols, int ylen, int grid, int sms)
{
    if (cols <= 0 || ylen <= 0) return 1;
    const long long items8 = cols * ((ylen + 7) / 8);
    if (items8 >= 4LL * grid) return (int)std::max<long long>(8, cols * ylen / (8LL * grid));
    if (items8 >= grid) {
        const long long n = 4LL * grid / cols;
        return (int)std::max<long long>(5, (ylen + n - 1) / n);
    }
    long long best = -1;
    int cy = ylen;
    for (int n = (ylen + 23) / 24; n <= std::max(1, ylen / 8); n++) {
        const int c = (ylen + n - 1) / n;
        const long long items = cols * ((ylen + c - 1) / c);
        const long long cost = (c + 7) * std::max<long long>(3, (items + sms - 1) / sms);
        if (best < 0 || cost <= best) {
            best = cost;
            cy = c;
        }
    }
    return cy;
}

// Planes a chunk of a launch, from the boxes of its shots.
int launch_chunk(const Grid &g, const Batch &b, int mode, int step, int grid)
{
    long long cols = 0;
    int ylen = 0;
    for (int s = 0; s < b.nshot; s++) {
        int lo[3], hi[3];
        box_bounds(g, (mode == s3::ADJ ? b.h_box_rec : b.h_box_src) + 6 * s, step, lo, hi);
        if (mode == s3::REC)
            for (int a = 0; a < 3; a++) {
                lo[a] = std::max(lo[a], g.L[a]);
                hi[a] = std::min(hi[a], g.H[a]);
            }
        if (hi[0] < lo[0] || hi[1] < lo[1]) continue;
        int base, rows;
        s3::tile_rows(lo[0], hi[0], base, rows);
        cols += (long long)rows * ((hi[1] - lo[1]) / s3::TX + 1);
        ylen = std::max(ylen, hi[2] - lo[2] + 1);
    }
    static const int sms = [] {
        int dev = 0, n = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
        return std::max(1, n);
    }();
    return pick_chunk(cols, ylen, grid, sms);
}

template <int N, int MODE>
void run_v(const LaunchCtx &lc, const Maps3 &m, const Grid &g, const Batch &b, const Fields &f, int step, const Gather3 &ga,
           const Restore3 &rs, unsigned *amax, unsigned *err, unsigned *ctr)
{
    constexpr int smem = s3::VLay<N, MODE>::SMEM;
    constexpr bool M = MODE == s3::FWD;
    auto *kernel = amax ? s3::k3_v<N, MODE, M> : s3::k3_v<N, MODE, false>;
    static const int grid = std::min(grid_for(s3::k3_v<N, MODE, M>, smem), grid_for(s3::k3_v<N, MODE, false>, smem));
    const s3::VMaps tm{m.p_halo, m.rho_v, m.vz_core, m.vx_core, m.vy_core, m.ezl_p, m.ezh_p, m.exl_p, m.exh_p};
    launch_pdl(lc, kernel, dim3(grid), s3::NTHR, smem, tm, g, b, f, step, launch_chunk(g, b, MODE, step, grid), ga,
               rs, amax, err, ctr);
}

template <int N, int MODE>
void run_p(const LaunchCtx &lc, const Maps3 &m, const Maps3 *lpm, const Grid &g, const Batch &b, const Fields &f, int step,
           unsigned *err, float *acc, int img_mode, const float *stf, float src_scale, const Save3 &sv, unsigned *ctr)
{
    constexpr int smem = s3::PLay<N, MODE>::SMEM;
    static const int grid = grid_for(s3::k3_p<N, MODE>, smem);
    const s3::PMaps tm{m.vz_halo, m.vx_halo, m.vy_core, m.p_core, m.K_core, lpm ? lpm->p_core : m.p_core,
                       m.ezl_v, m.ezh_v, m.exl_v, m.exh_v};
    launch_pdl(lc, s3::k3_p<N, MODE>, dim3(grid), s3::NTHR, smem, tm, g, b, f, step,
               launch_chunk(g, b, MODE, step, grid), err, acc, img_mode, stf, src_scale, sv, ctr);
}

}  // namespace

bool make_tile_map(CUtensorMap *tm, const Grid &g, const float *base, int nshot, int bz, int bx)
{
    return make_map(tm, g, base, nshot, bz, bx);
}

bool tile_maps_available() { return encoder() != nullptr; }

// The 3D path indexes one shot's arrays with 32-bit offsets.
void launch_wait_check(const LaunchCtx &lc, unsigned *err, long long polls)
{
    s3::k_wait_check<<<1, 32, 0, static_cast<cudaStream_t>(lc.stream)>>>(err, polls);
    ++*lc.launches;
}

long long wait_polls_default() { return s3::kSpin; }

bool stencil3d_supported(const Grid &g)
{
    return g.ndim == 3 && (g.N == 2 || g.N == 4) && g.ntot < (1LL << 31) && encoder() != nullptr;
}

bool make_maps3(Maps3 &m, const Grid &g, const Fields &f, int nshot, bool slabs)
{
    const int R = s3::TX + 2 * g.N - 1;
    Grid gr = g;                              // rho: the row padding repeats the last node (k_extend_model)
    gr.ne[0] = g.px;
    bool ok = make_map(&m.p_halo, g, f.p, nshot, s3::ZW, R) && make_map(&m.p_core, g, f.p, nshot, s3::TZ, s3::TX) &&
              make_map(&m.vz_core, g, f.v[0], nshot, s3::TZ, s3::TX) &&
              make_map(&m.vx_core, g, f.v[1], nshot, s3::TZ, s3::TX) &&
              make_map(&m.vy_core, g, f.v[2], nshot, s3::TZ, s3::TX) &&
              make_map(&m.vz_halo, g, f.v[0], nshot, s3::ZW, s3::TX) &&
              make_map(&m.vx_halo, g, f.v[1], nshot, s3::TZ, R) &&
              make_map(&m.rho_v, gr, g.rho, 1, 36, s3::TX + 1) && make_map(&m.K_core, g, g.K, 1, s3::TZ, s3::TX);
    if (!ok) return false;
    if (!slabs) {
        m.ezl_p = m.ezh_p = m.exl_p = m.exh_p = m.ezl_v = m.ezh_v = m.exl_v = m.exh_v = m.p_core;   // never read
        return true;
    }
    // z slab arrays [y][x][zp]: low and high part; x slab arrays [y][row][px]
    auto zmap = [&](CUtensorMap *lo, CUtensorMap *hi, const float *a) {
        const int nhi = g.zp - g.zlo;
        return make_slab_map(lo, a, g.zlo, g.ne[1], g.ne[2], nshot, g.zp, (long long)g.zp * g.ne[1], g.slab_n[0], s3::ZW,
                             s3::TX) &&
               (nhi > 0 ? make_slab_map(hi, a + g.zlo, nhi, g.ne[1], g.ne[2], nshot, g.zp, (long long)g.zp * g.ne[1],
                                        g.slab_n[0], s3::ZW, s3::TX)
                        : (*hi = *lo, true));
    };
    auto xmap = [&](CUtensorMap *lo, CUtensorMap *hi, const float *a) {
        const int nhi = g.xrows - g.xlo;
        return make_slab_map(lo, a, g.px, g.xlo, g.ne[2], nshot, g.px, (long long)g.px * g.xrows, g.slab_n[1], s3::TZ, R) &&
               (nhi > 0 ? make_slab_map(hi, a + (long long)g.xlo * g.px, g.px, nhi, g.ne[2], nshot, g.px,
                                        (long long)g.px * g.xrows, g.slab_n[1], s3::TZ, R)
                        : (*hi = *lo, true));
    };
    return zmap(&m.ezl_p, &m.ezh_p, f.psiv[0]) && xmap(&m.exl_p, &m.exh_p, f.psiv[1]) &&
           zmap(&m.ezl_v, &m.ezh_v, f.psip[0]) && xmap(&m.exl_v, &m.exh_v, f.psip[1]);
}

void launch3_v(const LaunchCtx &lc, const Maps3 &m, const Grid &g, const Batch &b, Fields f, int step, int mode,
               Gather3 ga, Restore3 rs, unsigned *amax, unsigned *err, unsigned *ctr)
{
    if (g.N == 2) {
        if (mode == 0) run_v<2, 0>(lc, m, g, b, f, step, ga, rs, amax, err, ctr);
        else if (mode == 1) run_v<2, 1>(lc, m, g, b, f, step, ga, rs, amax, err, ctr);
        else run_v<2, 2>(lc, m, g, b, f, step, ga, rs, amax, err, ctr);
    } else {
        if (mode == 0) run_v<4, 0>(lc, m, g, b, f, step, ga, rs, amax, err, ctr);
        else if (mode == 1) run_v<4, 1>(lc, m, g, b, f, step, ga, rs, amax, err, ctr);
        else run_v<4, 2>(lc, m, g, b, f, step, ga, rs, amax, err, ctr);
    }
}

void launch3_p(const LaunchCtx &lc, const Maps3 &m, const Maps3 *lpm, const Grid &g, const Batch &b, Fields f,
               int step, int mode, unsigned *err, float *acc, int img_mode, const float *stf, float src_scale, Save3 sv,
               unsigned *ctr)
{
    if (g.N == 2) {
        if (mode == 0) run_p<2, 0>(lc, m, lpm, g, b, f, step, err, acc, img_mode, stf, src_scale, sv, ctr);
        else if (mode == 1) run_p<2, 1>(lc, m, lpm, g, b, f, step, err, acc, img_mode, stf, src_scale, sv, ctr);
        else run_p<2, 2>(lc, m, lpm, g, b, f, step, err, acc, img_mode, stf, src_scale, sv, ctr);
    } else {
        if (mode == 0) run_p<4, 0>(lc, m, lpm, g, b, f, step, err, acc, img_mode, stf, src_scale, sv, ctr);
        else if (mode == 1) run_p<4, 1>(lc, m, lpm, g, b, f, step, err, acc, img_mode, stf, src_scale, sv, ctr);
        else run_p<4, 2>(lc, m, lpm, g, b, f, step, err, acc, img_mode, stf, src_scale, sv, ctr);
    }
}

}  // namespace smi
