// smi_stencil2d.cu -- 2D time steps in one launch each (sm_103a).
//
// A leap-frog step (Sec. 2.1 update equations) updates the velocities from
// the pressure and then the pressure from them.  One launch does both: a
// block takes a tile of 32 (z) x TX (x) nodes, brings the pressure with the
// halo of the whole step (2N - 1 nodes) by TMA into shared memory, computes
// the velocities of its nodes and of the N halo nodes its pressure update
// reads (1.2 - 1.4 times the tile), keeps them in shared memory, and updates
// the pressure from there.  Because a neighbour recomputes the same halo
// velocities from the old state, every step reads one set of arrays and
// writes the other (c -> n, swapped by the caller).  Kernels:
//   k2_fwd  forward step with the CPML memory variables (Komatitsch &
//           Martin), the source, boundary saving (Sec. 4.2) of the velocities
//           before the step, and the receivers' samples of the pressure
//           before the step (extra blocks);
//   k2_rev  one reverse step of Algorithm 2: blocks of even blockIdx.z take
//           the exact discrete adjoint in "same solver" form on the box of
//           the receivers (operands q + e, see smi_slab.h), blocks of odd z
//           the reconstruction of the source field backwards in time on the
//           physical domain -- pressure first, then the velocities, whose
//           boundary band comes from the store -- fused with the imaging /
//           gradient accumulation.  Both read only the old states, so they
//           share the launch.
//
// Why: the problem's fields are small (0.2 - 1.5 MB a shot), so a step is
// bound by launches and by the latency of a short chain of loads, or, with
// many shots, by issue and L2 traffic; one pass moves 24 B a point where a
// velocity and a pressure pass move 36, and a step is one launch instead of
// four to nine.  Against the two-pass kernels with their own launches for
// sources, receivers and bands (GB300): 201 x 201 order 4 forward, one shot,
// 16.9 -> 3.2 us a step; 257 x 903 order 8 gradient, one shot, 16-bit
// boundaries, 69.5 -> 14.6 us a step pair; 301 x 1001, 40 shots, 315 -> 165.
// Most tiles of a survey meet no slab, box edge, band or source: they run a
// body without tests or memory variables, in packed pairs (40 shots, whole
// grid: forward 172 -> 153 us, reverse 353 -> 273).
//
// Rows are padded to px (a multiple of 8), the padding of the fields holds
// zeros and TMA fills zeros outside the grid: the scheme's zero values.
// Offsets inside one shot's arrays are 32-bit (fewer than 2^31 points).
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <algorithm>

#include "smi_band.h"
#include "smi_box.h"
#include "smi_internal.h"
#include "smi_pack.h"
#include "smi_pdl.h"
#include "smi_slab.h"
#include "smi_stencil2d.h"
#include "smi_stencil3d.h"
#include "smi_tile3d.h"

namespace smi {

namespace {

using s3::in_range;
using s3::mbar_expect;
using s3::mbar_fence_init;
using s3::mbar_init;
using s3::mbar_wait;
using s3::put;
using s3::tma4;

// Tile widths and register budgets, by the 32 x 32 tiles of a launch over the
// whole grid (all shots).  Below kMany a launch hardly fills the GPU: narrow
// tiles (more, shorter blocks) and the registers a thread wants (4 blocks of
// 128 threads a SM, no spills).  Above, the blocks hide each other's load
// phases: forward 6 narrow blocks a SM (80 registers, 60 - 160 bytes spilled),
// reverse 4 wide ones (64 registers, 0.4 KB spilled).  Measured (us a step, or a step pair): forward 201 x 601, 4
// shots, order 8: narrow 4.3, narrow with 6 blocks 4.9, wide 5.2; 40 shots
// 301 x 1001 gradient with the forward narrow / 4 blocks 172, narrow / 6 166,
// wide / 3 169, and the reverse wide / 3 175, wide / 4 165, wide / 5 174, narrow
// 211; reverse at 8 shots 201 x 601 (1344 tiles) wide 17.7, narrow 18.6, at 4
// shots wide 12.5, narrow 12.1.
constexpr int kMany = 1200;
constexpr int kFwdTX = 16;
constexpr int kMaxRows = 65535;    // gridDim.y of a launch: longer models take several a step
constexpr int kRevBlocks = 4;

enum { FWD = 0, ADJ = 1 };

// Shared tiles (floats).  Forward / adjoint: pressure rows x0-2N+1 ..
// x0+TX+2N-2, z0-8 .. z0+39; v_z operand z0-4 .. z0+35 on the own rows; v_x
// operand on the own z, rows x0-N .. x0+TX+N-2.  Reconstruction: v_z and v_x
// with the halo of the pressures it recomputes, then those pressures.
template <int N, int TX> struct Lay {
    static constexpr int PW = 48, VW = 40;
    static constexpr int PR = TX + 4 * N - 2, XR = TX + 2 * N - 1;
    static constexpr int P = PW * PR, VZ = VW * TX, VX = 32 * XR;
    static constexpr int FA = P + VZ + VX;
    static constexpr int RZB = PW * XR, RXB = VW * PR;          // copied by TMA
    static constexpr int RZ = s3::rup32(RZB), RX = s3::rup32(RXB), RP = VW * XR;
    static constexpr int REC = RZ + RX + RP;
    static constexpr int MAXF = FA > REC ? FA : REC;
};

// rho of the quad one node up the z axis from r0 = rho of the quad (the row
// padding repeats the last node: 2 / (rho + rho) = 1 / rho there).
__device__ __forceinline__ Q4 rho_up(const Grid &g, int oz, int k, const Q4 &r0)
{
    float a[4];
    split(r0, a);
    return quad({a[1], a[2], a[3], oz + 4 < g.px ? g.rho[k + 4] : a[3]});
}
// v where the quad's nodes lie in [lo, hi] along z (and x in), else 0.
__device__ __forceinline__ Q4 masked(float v, int oz, bool x_in, int lo, int hi)
{
    float a[4];
#pragma unroll
    for (int r = 0; r < 4; r++) a[r] = x_in && in_range(oz + r, lo, hi) ? v : 0.0f;
    return quad(a);
}
// CPML coefficients of a quad along z, 0 where m is 0.
__device__ __forceinline__ void zcoefs(const float *tab, int oz, const Q4 &m, float (&c)[4])
{
    float a[4];
    split(m, a);
    put(c, s3::ldg4(tab + oz));
#pragma unroll
    for (int r = 0; r < 4; r++) c[r] = a[r] != 0.0f ? c[r] : 0.0f;
}
__device__ __forceinline__ void xcoefs(float v, const Q4 &m, float (&c)[4])
{
    float a[4];
    split(m, a);
#pragma unroll
    for (int r = 0; r < 4; r++) c[r] = a[r] != 0.0f ? v : 0.0f;
}
// v - b D (forward) or, b negative, v + b D (adjoint).
template <int MODE> __device__ __forceinline__ Q4 update(const Q4 &v, const Q4 &b, const Q4 &D)
{
    if (MODE == FWD) {
        float x[4], c[4], d[4];
        split(v, x);
        split(b, c);
        split(D, d);
#pragma unroll
        for (int r = 0; r < 4; r++) x[r] = __fmaf_rn(-c[r], d[r], x[r]);
        return quad(x);
    }
    return fmaq(b, D, v);
}

// The block's share of a step.
struct Tile {
    int s, z0, x0;
    int lo[3], hi[3];
};

struct SrcBox {
    int f0, f1, n0, n1;
};
__device__ __forceinline__ SrcBox src_box(const Batch &b, int s)
{
    const Stencil &st = b.src[s];
    return {st.first[0], st.first[1], st.cnt[0], st.cnt[1]};
}
// Whether the stencil meets nodes [z0, z1] x [x0, x1].
__device__ __forceinline__ bool src_near(const SrcBox &sb, int z0, int z1, int x0, int x1)
{
    return sb.f0 <= z1 && sb.f0 + sb.n0 - 1 >= z0 && sb.f1 <= x1 && sb.f1 + sb.n1 - 1 >= x0;
}
__device__ __forceinline__ void add_source(const Batch &b, const SrcBox &sb, int s, int oz, int ox, float amp, Q4 &q)
{
    const int t1 = ox - sb.f1;
    if (t1 < 0 || t1 >= sb.n1 || oz + 3 < sb.f0 || oz >= sb.f0 + sb.n0) return;
    float p[4];
    split(q, p);
    const Stencil &st = b.src[s];
#pragma unroll
    for (int r = 0; r < 4; r++) {
        const int t0 = oz + r - sb.f0;
        if (t0 >= 0 && t0 < sb.n0) p[r] += amp * st.w[0][t0] * st.w[1][t1] * st.w[2][0];
    }
    q = quad(p);
}

// Where the quad at (oz, ox) meets the boundary regions: bit r of z[sd] for
// node r in the z band of side sd (2N - 1 half nodes across the face, over the
// physical x), xs = side of the x band that holds the column (-1: none) with
// bit r of x for the physical z; and the offsets of node 0 in the stored step.
template <int N> struct BandQuad {
    unsigned z[2], x;
    int xs, zo[2], xo;
    __device__ __forceinline__ BandQuad(const Grid &g, const Bands &bd, int oz, int ox, bool own)
    {
        constexpr unsigned W = 2 * N - 2;              // last index across a face
        const bool px = own && in_range(ox, g.L[1], g.H[1]);
        const int t0 = oz - (g.L[0] - N), t1 = oz - (g.H[0] - N + 1);
        const unsigned u0 = (unsigned)(ox - (g.L[1] - N)), u1 = (unsigned)(ox - (g.H[1] - N + 1));
        z[0] = z[1] = x = 0u;
#pragma unroll
        for (int r = 0; r < 4; r++) {
            z[0] |= (px && (unsigned)(t0 + r) <= W) ? 1u << r : 0u;
            z[1] |= (px && (unsigned)(t1 + r) <= W) ? 1u << r : 0u;
            x |= (own && in_range(oz + r, g.L[0], g.H[0])) ? 1u << r : 0u;
        }
        xs = u0 <= W ? 0 : (u1 <= W ? 1 : -1);
        if (xs < 0) x = 0u;
        zo[0] = (int)bd.off[0][0] + t0 + (int)(W + 1) * (ox - g.L[1]);
        zo[1] = (int)bd.off[0][1] + t1 + (int)(W + 1) * (ox - g.L[1]);
        xo = (int)(xs == 1 ? bd.off[1][1] : bd.off[1][0]) + (oz - g.L[0]) +
             (g.H[0] - g.L[0] + 1) * (int)(xs == 1 ? u1 : u0);
    }
};
// Whether the block's own nodes meet a band of either axis (uniform).
template <int TX> __device__ __forceinline__ bool band_tile(const Bands &bd, int z0, int x0)
{
    bool m = false;
#pragma unroll
    for (int a = 0; a < 2; a++)
#pragma unroll
        for (int sd = 0; sd < 2; sd++)
            m = m || (z0 <= bd.hi[a][sd][0] && z0 + 31 >= bd.lo[a][sd][0] && x0 <= bd.hi[a][sd][1] &&
                      x0 + TX - 1 >= bd.lo[a][sd][1]);
    return m;
}

// 16-bit storage is scaled per (step, axis, side): the largest magnitude
// maps to 2^14 (FP16) or 1 (BF16).  Stores the quad's nodes in mask at
// o .. o+3 of the step that starts at base.
__device__ __forceinline__ void band_store(const Bands &bd, float scale, long long base, int o, unsigned mask, const Q4 &q)
{
    float v[4];
    split(q, v);
    if (bd.prec == SMI_PREC_F32) {
        float *d = static_cast<float *>(bd.data) + base + o;
#pragma unroll
        for (int r = 0; r < 4; r++)
            if (mask >> r & 1u) d[r] = v[r];
        return;
    }
    // one reciprocal a quad; early steps, whose scale is so small that it would overflow, divide
    const bool tiny = scale < 1e-36f;
    const float inv = tiny ? 0.0f : __frcp_rn(scale);
#pragma unroll
    for (int r = 0; r < 4; r++) {
        if (!(mask >> r & 1u)) continue;
        float y = v[r] * inv;
        if (tiny) y = scale > 0.0f ? v[r] / scale : 0.0f;
        if (bd.prec == SMI_PREC_F16) static_cast<__half *>(bd.data)[base + o + r] = __float2half_rn(y);
        else static_cast<__nv_bfloat16 *>(bd.data)[base + o + r] = __float2bfloat16_rn(y);
    }
}
// The stored values into the quad's nodes in mask, 0 where keep lacks them.
__device__ __forceinline__ void band_restore(const Bands &bd, float scale, long long base, int o, unsigned mask, unsigned keep,
                                             Q4 &q)
{
    float v[4];
    split(q, v);
#pragma unroll
    for (int r = 0; r < 4; r++)
        if (mask >> r & 1u) v[r] = keep >> r & 1u ? band_load(bd, base + o + r, scale) : 0.0f;
    q = quad(v);
}
// One velocity quad: v -+ b D, the memory variable m of the v grid (B, A: its
// coefficients), and the operand that the pressure update differentiates
// (forward: v; adjoint: v + e), returned.
template <int MODE>
__device__ __forceinline__ Q4 vel_quad(const Q4 &b, Q4 D, bool slab, const float (&B)[4], const float (&A)[4], float (&m)[4],
                                       Q4 &v)
{
    if (MODE == FWD && slab) {
        recur4(B, A, m, D);
        D = addq(D, quad(m));
    }
    v = update<MODE>(v, b, D);
    if (MODE == ADJ && slab) {
        recur4(B, A, m, v);
        return addq(v, quad(m));
    }
    return v;
}

// Forward or adjoint step of one tile.  sm: the block's shared tiles.  FAST:
// a tile whose nodes and halo lie inside the box and away from the slabs, the
// free surface, the source and the bands (tile_fast): no tests, no memory
// variables.
template <int N, int MODE, int TX, bool FAST, bool SAVE>
__device__ __forceinline__ void tile_step(const CUtensorMap *tm_p, const Grid &g, const Batch &b, const Fields &c,
                                          const Fields &n, const Tile &t, int step, const float *stf, float src_scale,
                                          const Bands &bd, const Save2 &save, const float *inj, float *sm,
                                          uint64_t *bar, unsigned *err)
{
    using La = Lay<N, TX>;
    constexpr int HX = 2 * N - 1, NT = 8 * TX;
    float *sp = sm, *svz = sm + La::P, *svx = svz + La::VZ;
    const int tid = threadIdx.x, tzi = tid & 7, txi = tid >> 3;
    const int s = t.s, z0 = t.z0, x0 = t.x0;
    const int oz = z0 + 4 * tzi, ox = x0 + txi, k = oz + g.px * ox;
    const bool own = FAST || (oz < g.ne[0] && ox < g.ne[1]);
    const long long sh = (long long)s * g.ntot;
    const long long so0 = (long long)s * g.slab_n[0], so1 = (long long)s * g.slab_n[1];
    const float dt2 = MODE == ADJ ? -2.0f * g.dt : 2.0f * g.dt;

    // extra velocity quads of the halo: threads below 2 TX take v_z on either
    // side along z, the next 8 (2N - 1) take v_x on either side along x
    int ez = 0, ex = 0;
    const bool exz = tid < 2 * TX;
    bool extra = exz;
    if (exz) {
        ez = (tid & 1) ? z0 + 32 : z0 - 4;
        ex = x0 + (tid >> 1);
    } else if (tid < 2 * TX + 8 * HX) {
        const int e = tid - 2 * TX, rr = e >> 3;
        ez = z0 + 4 * (e & 7);
        ex = rr < N ? x0 - N + rr : x0 + TX + rr - N;
        extra = true;
    }
    const bool ein = extra && (FAST || (ez >= 0 && ez < g.ne[0] && ex >= 0 && ex < g.ne[1]));
    const int ke = ez + g.px * ex;

    // ---- what no earlier step writes: model, coefficients, source stencil ----
    // buoyancies: 2 dt / (rho + rho') at the nodes of the box, else 0
    const Q4 two = quad({dt2, dt2, dt2, dt2});
    Q4 in = two, ie = two;
    if (!FAST) {
        in = masked(dt2, oz, own && in_range(ox, t.lo[1], t.hi[1]), t.lo[0], t.hi[0]);
        ie = masked(dt2, ez, ein && in_range(ex, t.lo[1], t.hi[1]), t.lo[0], t.hi[0]);
    }
    Q4 bz = zeroq(), bx = zeroq(), be = zeroq(), Kv = zeroq();
    if (own) {
        const Q4 r0 = ldq(g.rho + k);
        bz = buoyq(in, r0, rho_up(g, oz, k, r0));
        bx = buoyq(in, r0, FAST || ox + 1 < g.ne[1] ? ldq(g.rho + k + g.px) : r0);
        Kv = ldq(g.K + k);
    }
    if (ein) {
        const Q4 r0 = ldq(g.rho + ke);
        be = buoyq(ie, r0, exz ? rho_up(g, ez, ke, r0) : (FAST || ex + 1 < g.ne[1] ? ldq(g.rho + ke + g.px) : r0));
    }
    const int zq = !FAST && own ? zslab_quad(g, oz) : -1, xq = !FAST && own ? slab_row(g, 1, ox) : -1;
    const int eq = !FAST && ein ? (exz ? zslab_quad(g, ez) : slab_row(g, 1, ex)) : -1;
    const long long zo = so0 + zq + (long long)g.zp * ox, xo = so1 + (long long)g.px * xq + oz;
    const long long eo = exz ? so0 + eq + (long long)g.zp * ex : so1 + (long long)g.px * eq + ez;
    SrcBox sb{0, 0, 0, 0};
    float amp = 0.0f;
    if (!FAST && MODE == FWD && stf) {
        sb = src_box(b, s);
        amp = src_scale * stf[step];
    }

    if (MODE == FWD) {                        // (the reverse kernel has waited)
        pdl_wait();
        pdl_trigger();
    }
    if (tid == 0) {
        mbar_expect(bar, (unsigned)La::P * 4u);
        tma4(sp, tm_p, z0 - 8, x0 - HX, 0, s, bar);
    }
    // ---- the old state ----
    Q4 vz = zeroq(), vx = zeroq(), ve = zeroq();
    float mz[4] = {}, mx[4] = {}, me[4] = {}, pz[4] = {}, px[4] = {};
    if (own) {
        vz = ldq(c.v[0] + sh + k);
        vx = ldq(c.v[1] + sh + k);
    }
    if (ein) ve = ldq((exz ? c.v[0] : c.v[1]) + sh + ke);
    if (!FAST) {
        if (zq >= 0) {
            put(mz, s3::ldg4(c.psip[0] + zo));
            put(pz, s3::ldg4(c.psiv[0] + zo));
        }
        if (xq >= 0) {
            put(mx, s3::ldg4(c.psip[1] + xo));
            put(px, s3::ldg4(c.psiv[1] + xo));
        }
        if (eq >= 0) put(me, s3::ldg4((exz ? c.psip[0] : c.psip[1]) + eo));
    }

    // scales of the sample this step stores (at the end, from the old arrays)
    const bool saves = !FAST && SAVE && save.sample >= 0 && band_tile<TX>(bd, z0, x0);
    float scale[4] = {0.0f, 0.0f, 0.0f, 0.0f};
    if (SAVE && save.sample >= 0 && bd.prec != SMI_PREC_F32) {
        const bool first = t.z0 == (t.lo[0] & ~3) && t.x0 == t.lo[1];      // writes the shot's scales
        if (saves || first) {
#pragma unroll
            for (int q = 0; q < 4; q++) {
                scale[q] = __uint_as_float(save.amax[((long long)save.sample * b.nshot + s) * 6 + q]) /
                           (bd.prec == SMI_PREC_F16 ? 16384.0f : 1.0f);
                if (first && tid == q) bd.scale[((long long)s * bd.nt + save.sample) * 6 + q] = scale[q];
            }
        }
    }

    if (!mbar_wait(bar, 0)) {                 // every thread gives up alike after the same number of polls
        if (tid == 0) atomicOr(err, 1u);
        mbar_wait(bar, 0);
    }
    float *const pz_own = svz + txi * La::VW + 4 * tzi + 4, *const px_own = svx + (txi + N) * 32 + 4 * tzi;

    // ---- velocities: own quads, then the halo's ----
    auto z_deriv = [&](int qz, int qx) {
        float W[12];
        window(W, sp + (qx - x0 + HX) * La::PW + (qz - z0) + 4);
        if (!FAST && MODE == ADJ && (qz - 4 < g.zlo || qz + 7 >= g.zhi) && qx >= 0 && qx < g.ne[1]) {
#pragma unroll
            for (int q = 0; q < 3; q++) {
                const int e = zslab_quad(g, qz - 4 + 4 * q);
                if (e < 0) continue;
                float a[4];
                put(a, s3::ldg4(c.psiv[0] + so0 + e + (long long)g.zp * qx));
#pragma unroll
                for (int r = 0; r < 4; r++) W[4 * q + r] += a[r];
            }
        }
        return dz4<N, true>(g, W);
    };
    auto x_deriv = [&](int qz, int qx) {
        Q4 D = zeroq();
        const bool near = !FAST && MODE == ADJ && (qx - N + 1 < g.xlo || qx + N >= g.xhi) && qz < g.ne[0];
        const float *row = sp + (qx - x0 + HX) * La::PW + (qz - z0) + 8;
#pragma unroll
        for (int l = 1; l <= N; l++) {
            Q4 a = ldq(row + l * La::PW), d = ldq(row - (l - 1) * La::PW);
            if (near) {
                const int ja = slab_row(g, 1, qx + l), jd = slab_row(g, 1, qx - l + 1);
                if (ja >= 0) a = addq(a, ldq(c.psiv[1] + so1 + (long long)g.px * ja + qz));
                if (jd >= 0) d = addq(d, ldq(c.psiv[1] + so1 + (long long)g.px * jd + qz));
            }
            D = tap(D, g.c[1][l - 1], a, d);
        }
        return D;
    };
    {
        float B[4] = {}, A[4] = {};
        if (!FAST && zq >= 0) {
            zcoefs(g.cvb[0], oz, in, B);
            zcoefs(g.cva[0], oz, in, A);
        }
        stq(pz_own, vel_quad<MODE>(bz, z_deriv(oz, ox), zq >= 0, B, A, mz, vz));
        if (!FAST && xq >= 0) {
            xcoefs(g.cvb[1][ox], in, B);
            xcoefs(g.cva[1][ox], in, A);
        }
        stq(px_own, vel_quad<MODE>(bx, x_deriv(oz, ox), xq >= 0, B, A, mx, vx));
    }
    if (extra) {
        float B[4] = {}, A[4] = {};
        float *const pe = exz ? svz + (ex - x0) * La::VW + (ez - z0 + 4) : svx + (ex - x0 + N) * 32 + (ez - z0);
        if (exz) {
            if (!FAST && eq >= 0) {
                zcoefs(g.cvb[0], ez, ie, B);
                zcoefs(g.cva[0], ez, ie, A);
            }
            stq(pe, vel_quad<MODE>(be, z_deriv(ez, ex), eq >= 0, B, A, me, ve));
        } else {
            if (!FAST && eq >= 0) {
                xcoefs(g.cvb[1][ex], ie, B);
                xcoefs(g.cva[1][ex], ie, A);
            }
            stq(pe, vel_quad<MODE>(be, x_deriv(ez, ex), eq >= 0, B, A, me, ve));
        }
    }
    __syncthreads();
    if (!FAST && g.freesurf && z0 - 4 < g.L[0]) {
        // free surface (image method): half node L-1-j mirrors L+j; the adjoint folds it there.  A tile that
        // holds an image row or has it in its halo holds its mirror (pressures above the tile: run_fwd); the
        // memory variables of these rows are zero (no absorption at the top).
        const int L = g.L[0];
        for (int i = tid; i < TX * N; i += NT) {
            const int r = i / N, j = i % N, zi = L - 1 - j - (z0 - 4), zm = L + j - (z0 - 4);
            if (zi < 0 || zm >= La::VW) continue;
            float *row = svz + r * La::VW;
            if (MODE == FWD) {
                row[zi] = row[zm];
            } else {
                row[zm] += row[zi];
                row[zi] = 0.0f;
            }
        }
        __syncthreads();
        if (oz < L + N) vz = ldq(pz_own);
    }

    // ---- pressure ----
    Q4 pv = ldq(sp + (txi + HX) * La::PW + 4 * tzi + 8);
    {
        float W[12], B[4], A[4];
        window(W, svz + txi * La::VW + 4 * tzi);
        Q4 Dz = dz4<N, false>(g, W), Dx = zeroq();
#pragma unroll
        for (int l = 1; l <= N; l++)
            Dx = tap(Dx, g.c[1][l - 1], ldq(svx + (txi + N + l - 1) * 32 + 4 * tzi), ldq(svx + (txi + N - l) * 32 + 4 * tzi));
        if (!FAST && MODE == FWD && zq >= 0) {
            zcoefs(g.cpb[0], oz, in, B);
            zcoefs(g.cpa[0], oz, in, A);
            recur4(B, A, pz, Dz);
            Dz = addq(Dz, quad(pz));
        }
        if (!FAST && MODE == FWD && xq >= 0) {
            xcoefs(g.cpb[1][ox], in, B);
            xcoefs(g.cpa[1][ox], in, A);
            recur4(B, A, px, Dx);
            Dx = addq(Dx, quad(px));
        }
        const float sg = MODE == ADJ ? -g.dt : g.dt;
        const Q4 dts = FAST ? quad({sg, sg, sg, sg})
                            : masked(sg, oz, own && in_range(ox, t.lo[1], t.hi[1]), t.lo[0], t.hi[0]);
        pv = update<MODE>(pv, mulq(dts, Kv), addq(Dz, Dx));
        if (MODE == ADJ && inj) pv = fmaq(Kv, ldq(inj + txi * 32 + 4 * tzi), pv);   // the next step's adjoint source
        if (!FAST && MODE == ADJ && zq >= 0) {
            zcoefs(g.cpb[0], oz, in, B);
            zcoefs(g.cpa[0], oz, in, A);
            recur4(B, A, pz, pv);
        }
        if (!FAST && MODE == ADJ && xq >= 0) {
            xcoefs(g.cpb[1][ox], in, B);
            xcoefs(g.cpa[1][ox], in, A);
            recur4(B, A, px, pv);
        }
    }
    if (!FAST && MODE == FWD && stf) add_source(b, sb, s, oz, ox, amp, pv);
    if (!FAST && MODE == FWD && g.freesurf && z0 <= g.L[0] + N) {
        // p = 0 on the surface row L, -p mirrored above it (the own pressures of the tile's centre)
        stq(sp + (txi + HX) * La::PW + 4 * tzi + 8, pv);
        __syncthreads();
        const int L = g.L[0];
        float p4[4];
        split(pv, p4);
#pragma unroll
        for (int r = 0; r < 4; r++) {
            const int z = oz + r, zm = 2 * L - z - z0;
            if (z == L) p4[r] = 0.0f;
            else if (z < L && z >= L - N && zm < 32) p4[r] = -sp[(txi + HX) * La::PW + zm + 8];
        }
        pv = quad(p4);
    }
    if (own) {
        stq(n.v[0] + sh + k, vz);
        stq(n.v[1] + sh + k, vx);
        stq(n.p + sh + k, pv);
        if (!FAST && zq >= 0) {
            s3::stg4(n.psip[0] + zo, mz);
            s3::stg4(n.psiv[0] + zo, pz);
        }
        if (!FAST && xq >= 0) {
            s3::stg4(n.psip[1] + xo, mx);
            s3::stg4(n.psiv[1] + xo, px);
        }
    }
    if (!FAST && SAVE && (save.sample >= 0 || save.next >= 0) && band_tile<TX>(bd, z0, x0)) {
        const BandQuad<N> bq(g, bd, oz, ox, own);
        if (saves && (bq.z[0] | bq.z[1] | bq.x)) {
            const Q4 vz_old = ldq(c.v[0] + sh + k), vx_old = ldq(c.v[1] + sh + k);
            const long long base = ((long long)s * bd.nt + save.sample) * bd.count;
            if (bq.z[0]) band_store(bd, scale[0], base, bq.zo[0], bq.z[0], vz_old);
            if (bq.z[1]) band_store(bd, scale[1], base, bq.zo[1], bq.z[1], vz_old);
            if (bq.x) band_store(bd, bq.xs ? scale[3] : scale[2], base, bq.xo, bq.x, vx_old);
        }
        if (save.next >= 0) {
            // largest magnitude per (axis, side) of the velocities the next sample stores
            unsigned *am = save.amax + ((long long)save.next * b.nshot + s) * 6;
            const unsigned m0 = warp_max(vz, bq.z[0]), m1 = warp_max(vz, bq.z[1]);
            const unsigned m2 = warp_max(vx, bq.xs == 0 ? bq.x : 0u), m3 = warp_max(vx, bq.xs == 1 ? bq.x : 0u);
            if ((tid & 31) == 0) {
                if (m0) atomicMax(am, m0);
                if (m1) atomicMax(am + 1, m1);
                if (m2) atomicMax(am + 2, m2);
                if (m3) atomicMax(am + 3, m3);
            }
        }
    }
}

// Whether the tile and its halo lie inside the box of the step and away from
// every special case (uniform over the block).
template <int N, int MODE, int TX>
__device__ __forceinline__ bool tile_fast(const Grid &g, const Batch &b, const Tile &t, bool src, const Bands &bd, bool bands)
{
    const int zl = t.z0 - 8, zh = t.z0 + 39, xl = t.x0 - 2 * N + 1, xh = t.x0 + TX + 2 * N - 2;
    bool f = t.z0 - 4 >= t.lo[0] && t.z0 + 35 <= t.hi[0] && t.x0 - N >= t.lo[1] && t.x0 + TX + N - 2 <= t.hi[1] &&
             zl >= g.zlo && zh < g.zhi && xl >= g.xlo && xh < g.xhi && !(g.freesurf && t.z0 - 4 <= g.L[0] + N);
    if (MODE == FWD && f && src) f = !src_near(src_box(b, t.s), t.z0, t.z0 + 31, t.x0, t.x0 + TX - 1);
    return f && !(bands && band_tile<TX>(bd, t.z0, t.x0));
}

// SAVE: boundary saving (a call that reverses the field later).  Rows of
// blocks y0 .. y0 + gridDim.y - 1 of the step: ng of receivers, then tiles.
template <int N, int BLOCKS, bool SAVE>
__global__ void __launch_bounds__(8 * kFwdTX, BLOCKS)
k2_fwd(const __grid_constant__ CUtensorMap tm_p, Grid g, Batch b, Fields c, Fields n, int step, const float *stf,
       float src_scale, Bands bd, Save2 save, Gather2 ga, int ng, int y0, unsigned *err)
{
    constexpr int TX = kFwdTX;
    __shared__ __align__(128) float sm[Lay<N, TX>::FA];
    __shared__ __align__(8) uint64_t bar;
    Tile t;
    t.s = blockIdx.z;
    const int row = (int)blockIdx.y + y0;
    if (row < ng) {                // receivers: samples of the pressure before the step
        const int nr = b.rec_off[t.s + 1] - b.rec_off[t.s];
        const int r = (row * gridDim.x + blockIdx.x) * (8 * TX) + threadIdx.x;
        const bool have = r < nr;
        const Stencil &st = b.rec[b.rec_off[t.s] + (have ? r : 0)];
        const float *ps = c.p + t.s * g.ntot + (have ? st.first[0] + g.px * st.first[1] : 0);
        const int n0 = have ? st.cnt[0] : 0, n1 = have ? st.cnt[1] : 0;
        float w0[2 * N], w1[2 * N];
#pragma unroll
        for (int a = 0; a < 2 * N; a++) {
            w0[a] = a < n0 ? st.w[0][a] : 0.0f;
            w1[a] = a < n1 ? st.w[1][a] : 0.0f;
        }
        pdl_wait();
        pdl_trigger();
        if (!have) return;
        float sum = 0.0f;
        if (n0 == 2 * N && n1 == 2 * N) {      // every tap: four rows of loads in flight
#pragma unroll
            for (int h = 0; h < 2 * N; h += 4) {
                float x[4][2 * N];
#pragma unroll
                for (int a1 = 0; a1 < 4; a1++)
#pragma unroll
                    for (int a0 = 0; a0 < 2 * N; a0++) x[a1][a0] = ps[a0 + g.px * (h + a1)];
#pragma unroll
                for (int a1 = 0; a1 < 4; a1++)
#pragma unroll
                    for (int a0 = 0; a0 < 2 * N; a0++) sum += w0[a0] * w1[h + a1] * x[a1][a0];
            }
        } else {
#pragma unroll
            for (int a1 = 0; a1 < 2 * N; a1++)
#pragma unroll
                for (int a0 = 0; a0 < 2 * N; a0++)
                    if (a0 < n0 && a1 < n1) sum += w0[a0] * w1[a1] * ps[a0 + g.px * a1];
        }
        ga.seis[ga.off[t.s] + (long long)ga.it * nr + r] = sum;
        return;
    }
    box_at(b.tab_src, b.nt1, t.s, step, t.lo, t.hi);
    t.z0 = (t.lo[0] & ~3) + 32 * blockIdx.x;
    t.x0 = t.lo[1] + TX * (row - ng);
    if (t.z0 > t.hi[0] || t.x0 > t.hi[1]) {
        if (blockIdx.x + blockIdx.y + blockIdx.z == 0) pdl_wait();   // one block of a launch always waits
        return;
    }
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        mbar_fence_init();
    }
    __syncthreads();
    if (tile_fast<N, FWD, TX>(g, b, t, stf != nullptr, bd, SAVE && (save.sample >= 0 || save.next >= 0)))
        tile_step<N, FWD, TX, true, SAVE>(&tm_p, g, b, c, n, t, step, stf, src_scale, bd, save, nullptr, sm, &bar, err);
    else
        tile_step<N, FWD, TX, false, SAVE>(&tm_p, g, b, c, n, t, step, stf, src_scale, bd, save, nullptr, sm, &bar, err);
}

// Reconstruction of one tile.  Own nodes: the physical domain and the
// boundary bands inside the box of step it + 1 (so that nodes which left the
// box are written as zeros into both sets of arrays).  FAST: a tile whose
// nodes and halo lie inside the box of the step before, the range that every
// velocity component updates, and away from the source and the bands.
template <int N, int TX, bool FAST>
__device__ __forceinline__ void tile_rec(const CUtensorMap *tm_vz, const CUtensorMap *tm_vx, const Grid &g,
                                         const Batch &b, const Fields &c, const Fields &n, const Tile &t, const int (&lo)[2],
                                         const int (&hi)[2], const int (&plo)[3], const int (&phi)[3], int it,
                                         const float *lp, float *acc, int img_mode, const float *stf, float src_scale,
                                         const Bands &bd, bool restore, float *sm, uint64_t *bar, unsigned *err)
{
    using La = Lay<N, TX>;
    constexpr int HX = 2 * N - 1;
    float *tz = sm, *tx = sm + La::RZ, *spn = tx + La::RX;
    const int tid = threadIdx.x, tzi = tid & 7, txi = tid >> 3;
    const int s = t.s, z0 = t.z0, x0 = t.x0;
    const int oz = z0 + 4 * tzi, ox = x0 + txi, k = oz + g.px * ox;
    const bool own = FAST || (oz < g.ne[0] && ox < g.ne[1]);
    const long long sh = (long long)s * g.ntot;
    const float dt = g.dt;
    if (tid == 0) {
        mbar_expect(bar, (unsigned)(La::RZB + La::RXB) * 4u);
        tma4(tz, tm_vz, z0 - 8, x0 - N + 1, 0, s, bar);
        tma4(tx, tm_vx, z0 - 4, x0 - HX, 0, s, bar);
    }
    int ez = 0, ex = 0;                       // extra pressure quads of the halo
    bool extra = tid < 2 * TX;
    if (extra) {
        ez = (tid & 1) ? z0 + 32 : z0 - 4;
        ex = x0 + (tid >> 1);
    } else if (tid < 2 * TX + 8 * HX) {
        const int e = tid - 2 * TX, rr = e >> 3;
        ez = z0 + 4 * (e & 7);
        ex = rr < N - 1 ? x0 - N + 1 + rr : x0 + TX + rr - (N - 1);
        extra = true;
    }
    const bool ein = extra && (FAST || (ez >= 0 && ez < g.ne[0] && ex >= 0 && ex < g.ne[1]));
    const int ke = ez + g.px * ex;

    const Q4 one = quad({dt, dt, dt, dt}), two = quad({2.0f * dt, 2.0f * dt, 2.0f * dt, 2.0f * dt});
    // dt (or 2 dt) at the nodes that the pressure and each velocity component update, else 0
    const bool inx = FAST || in_range(ox, lo[1], hi[1]);
    const Q4 dp = FAST ? one : masked(dt, oz, inx, lo[0], hi[0]);
    const Q4 de = FAST ? one : masked(dt, ez, ein && in_range(ex, lo[1], hi[1]), lo[0], hi[0]);
    const Q4 dz = FAST ? two : masked(2.0f * dt, oz, inx, max(lo[0], g.L[0] + N - 1), min(hi[0], g.H[0] - N));
    const Q4 dx = FAST ? two : masked(2.0f * dt, oz, inx && in_range(ox, g.L[1] + N - 1, g.H[1] - N), lo[0], hi[0]);
    Q4 bz = zeroq(), bx = zeroq(), Kv = zeroq(), Ke = zeroq(), pv = zeroq(), pe = zeroq(), lpv = zeroq(), av = zeroq();
    if (own) {
        const Q4 r0 = ldq(g.rho + k);
        bz = buoyq(dz, r0, rho_up(g, oz, k, r0));
        bx = buoyq(dx, r0, FAST || ox + 1 < g.ne[1] ? ldq(g.rho + k + g.px) : r0);
        Kv = ldq(g.K + k);
        pv = ldq(c.p + sh + k);
        lpv = ldq(lp + sh + k);
        av = ldq(acc + sh + k);
    }
    if (ein) {
        Ke = ldq(g.K + ke);
        pe = ldq(c.p + sh + ke);
    }
    SrcBox sb{0, 0, 0, 0};
    float amp = 0.0f;
    if (!FAST) {
        sb = src_box(b, s);
        amp = -src_scale * stf[it];
    }
    const bool bands = !FAST && band_tile<TX>(bd, z0, x0);
    float scale[4] = {1.0f, 1.0f, 1.0f, 1.0f};
    if (!FAST && restore && bands && bd.prec != SMI_PREC_F32) {
#pragma unroll
        for (int q = 0; q < 4; q++) scale[q] = bd.scale[((long long)s * bd.nt + it) * 6 + q];
    }
    if (!mbar_wait(bar, 0)) {
        if (tid == 0) atomicOr(err, 1u);
        mbar_wait(bar, 0);
    }
    // nodes of the update region d (not 0) that the previous box leaves out
    auto clear_left = [&](Q4 &q, const Q4 &d, int qz, int qx) {
        float m[4];
        bool cl[4];
        split(d, m);
        const bool kx = in_range(qx, plo[1], phi[1]);
#pragma unroll
        for (int r = 0; r < 4; r++) cl[r] = m[r] != 0.0f && !(kx && in_range(qz + r, plo[0], phi[0]));
        q = clear_if(q, cl);
    };

    // ---- pressures: p + dt kappa div v - source, zero outside the previous box ----
    auto div_at = [&](int qz, int qx) {
        float W[12];
        window(W, tz + (qx - x0 + N - 1) * La::PW + (qz - z0) + 4);
        const Q4 Dz = dz4<N, false>(g, W);
        Q4 Dx = zeroq();
        const float *row = tx + (qx - x0 + HX) * La::VW + (qz - z0) + 4;
#pragma unroll
        for (int l = 1; l <= N; l++) Dx = tap(Dx, g.c[1][l - 1], ldq(row + (l - 1) * La::VW), ldq(row - l * La::VW));
        return addq(Dz, Dx);
    };
    auto press = [&](int qz, int qx, const Q4 &d, const Q4 &K4, const Q4 &p, const Q4 &dv) {
        Q4 q = fmaq(mulq(d, K4), dv, p);
        if (FAST) return q;
        Q4 w = q;
        add_source(b, sb, s, qz, qx, amp, w);
        float m[4], a[4], e[4];
        split(d, m);
        split(q, a);
        split(w, e);
#pragma unroll
        for (int r = 0; r < 4; r++) {
            if (m[r] != 0.0f) a[r] = e[r];
            if (m[r] != 0.0f && g.freesurf && qz + r == g.L[0]) a[r] = 0.0f;
        }
        q = quad(a);
        clear_left(q, d, qz, qx);
        return q;
    };
    {
        const Q4 dv = div_at(oz, ox), np = press(oz, ox, dp, Kv, pv, dv);
        stq(spn + (txi + N - 1) * La::VW + 4 * tzi + 4, np);
        if (own) {
            stq(n.p + sh + k, np);
            Q4 t = img_mode == 0 ? dv : pv;
            if (!FAST && img_mode == 0) {      // div v reaches past the box (p does not)
                float m[4];
                bool out[4];
                split(dp, m);
#pragma unroll
                for (int r = 0; r < 4; r++) out[r] = m[r] == 0.0f;
                t = clear_if(t, out);
            }
            stq(acc + sh + k, fmaq(lpv, t, av));
            if (img_mode == 2) {               // illumination
                float *ill = acc + (long long)b.nshot * g.ntot + sh + k;
                stq(ill, fmaq(pv, pv, ldq(ill)));
            }
        }
    }
    if (extra) stq(spn + (ex - x0 + N - 1) * La::VW + (ez - z0) + 4, press(ez, ex, de, Ke, pe, div_at(ez, ex)));
    Q4 vz = ldq(tz + (txi + N - 1) * La::PW + 4 * tzi + 8), vx = ldq(tx + (txi + HX) * La::VW + 4 * tzi + 4);
    __syncthreads();

    // ---- velocities: v_a + dt b_a D_a p on L_a+N-1 .. H_a-N, the bands from the store ----
    float W[12];
    window(W, spn + (txi + N - 1) * La::VW + 4 * tzi);
    const Q4 D = dz4<N, true>(g, W);
    Q4 X = zeroq();
#pragma unroll
    for (int l = 1; l <= N; l++)
        X = tap(X, g.c[1][l - 1], ldq(spn + (txi + N - 1 + l) * La::VW + 4 * tzi + 4),
                ldq(spn + (txi + N - l) * La::VW + 4 * tzi + 4));
    vz = fmaq(bz, D, vz);
    vx = fmaq(bx, X, vx);
    if (!FAST) {
        clear_left(vz, dz, oz, ox);
        clear_left(vx, dx, oz, ox);
        if (restore && bands) {                // zero (and not stored) outside the previous box
            const BandQuad<N> bq(g, bd, oz, ox, own);
            const long long base = ((long long)s * bd.nt + it) * bd.count;
            const bool kx = in_range(ox, plo[1], phi[1]);
            unsigned keep = 0u;
#pragma unroll
            for (int r = 0; r < 4; r++) keep |= kx && in_range(oz + r, plo[0], phi[0]) ? 1u << r : 0u;
            if (bq.z[0]) band_restore(bd, scale[0], base, bq.zo[0], bq.z[0], keep, vz);
            if (bq.z[1]) band_restore(bd, scale[1], base, bq.zo[1], bq.z[1], keep, vz);
            if (bq.x) band_restore(bd, bq.xs ? scale[3] : scale[2], base, bq.xo, bq.x, keep, vx);
        }
    }
    if (own) {
        stq(n.v[0] + sh + k, vz);
        stq(n.v[1] + sh + k, vx);
    }
}

// roles 1: adjoint, 2: reconstruction (blockIdx.z = shot), 3: both
// (blockIdx.z = 2 shot + role, 0 adjoint, 1 reconstruction).  Tile rows from y0.
template <int N, int TX>
__global__ void __launch_bounds__(8 * TX, kRevBlocks)
k2_rev(const __grid_constant__ CUtensorMap tm_lp, const __grid_constant__ CUtensorMap tm_vz,
       const __grid_constant__ CUtensorMap tm_vx, Grid g, Batch b, Fields ac, Fields an, int mrev, int roles, Fields fc,
       Fields fn, int it, float *acc, int img_mode, const float *stf, float src_scale, Bands bd, int restore,
       Inject2 ij, int y0, unsigned *err)
{
    __shared__ __align__(128) float sm[Lay<N, TX>::MAXF];
    __shared__ __align__(16) float sinj[32 * TX];
    __shared__ __align__(8) uint64_t bar;
    const bool role = roles == 3 ? blockIdx.z & 1 : roles == 2;
    Tile t;
    t.s = roles == 3 ? blockIdx.z >> 1 : blockIdx.z;
    if (role) {
        box_at(b.tab_src, b.nt1, t.s, min(it + 1, b.nt1 - 2), t.lo, t.hi);
#pragma unroll
        for (int a = 0; a < 2; a++) {
            t.lo[a] = max(t.lo[a], g.L[a] - N);
            t.hi[a] = min(t.hi[a], g.H[a] + N - 1);
        }
    } else {
        box_at(b.tab_rec, b.nt1, t.s, mrev, t.lo, t.hi);
    }
    t.z0 = (t.lo[0] & ~3) + 32 * blockIdx.x;
    t.x0 = t.lo[1] + TX * ((int)blockIdx.y + y0);
    if (t.z0 > t.hi[0] || t.x0 > t.hi[1]) {
        if (blockIdx.x + blockIdx.y + blockIdx.z == 0) pdl_wait();
        return;
    }
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        mbar_fence_init();
    }
    // The adjoint source of the reverse step after this one, sum over receivers of weight times residual at
    // the tile's nodes: it enters the adjoint pressure as this step writes it (nothing here is written by an
    // earlier step, so it is done before the wait).  Receivers are listed by cells of 32 columns.
    const float *inj = nullptr;
    if (!role && ij.it >= 0) {
        const int *e = b.box_rec + 6 * t.s;
        if (e[0] <= t.z0 + 31 && e[3] >= t.z0 && e[1] <= t.x0 + TX - 1 && e[4] >= t.x0) {
            for (int i = threadIdx.x; i < 32 * TX; i += 8 * TX) sinj[i] = 0.0f;
            __syncthreads();
            const int nr = b.rec_off[t.s + 1] - b.rec_off[t.s];
            const float *res = ij.res + ij.off[t.s] + (long long)ij.it * nr;
            const int c1 = min((t.x0 + TX - 1) >> 5, ij.ncell - 1);
            for (int c = t.x0 >> 5; c <= c1; c++) {
                const int *co = ij.cell + (long long)t.s * (ij.ncell + 1) + c;
                for (int i = co[0] + threadIdx.x; i < co[1]; i += 8 * TX) {
                    const int r = ij.ids[i];
                    const Stencil &st = b.rec[b.rec_off[t.s] + r];
                    const float val = res[r];
                    const int xa = max(st.first[1], max(t.x0, c << 5));
                    const int xb = min(st.first[1] + st.cnt[1] - 1, min(t.x0 + TX - 1, (c << 5) + 31));
                    const int za = max(st.first[0], t.z0), zb = min(st.first[0] + st.cnt[0] - 1, t.z0 + 31);
                    for (int x = xa; x <= xb; x++)
                        for (int z = za; z <= zb; z++)
                            atomicAdd(sinj + (x - t.x0) * 32 + z - t.z0,
                                      st.w[0][z - st.first[0]] * st.w[1][x - st.first[1]] * st.w[2][0] * val);
                }
            }
            inj = sinj;
        }
    }
    __syncthreads();
    pdl_wait();
    pdl_trigger();
    if (role) {
        // update region (box of the step within the physical domain), previous box
        int lo[2], hi[2], plo[3], phi[3], bl[3], bh[3];
        box_at(b.tab_src, b.nt1, t.s, it - 1, plo, phi);
        box_at(b.tab_src, b.nt1, t.s, it, bl, bh);
        bool fast = !band_tile<TX>(bd, t.z0, t.x0) &&
                    !src_near(src_box(b, t.s), t.z0 - 4, t.z0 + 35, t.x0 - N + 1, t.x0 + TX - 1 + N);
#pragma unroll
        for (int a = 0; a < 2; a++) {
            lo[a] = max(bl[a], g.L[a]);
            hi[a] = min(bh[a], g.H[a]);
            const int l = a == 0 ? t.z0 - 4 : t.x0 - N + 1, h = a == 0 ? t.z0 + 35 : t.x0 + TX - 1 + N;
            fast = fast && l >= max(lo[a], max(plo[a], g.L[a] + N - 1)) && h <= min(hi[a], min(phi[a], g.H[a] - N));
        }
        if (fast)
            tile_rec<N, TX, true>(&tm_vz, &tm_vx, g, b, fc, fn, t, lo, hi, plo, phi, it, ac.p, acc, img_mode, stf,
                                  src_scale, bd, restore != 0, sm, &bar, err);
        else
            tile_rec<N, TX, false>(&tm_vz, &tm_vx, g, b, fc, fn, t, lo, hi, plo, phi, it, ac.p, acc, img_mode, stf,
                                   src_scale, bd, restore != 0, sm, &bar, err);
    } else if (tile_fast<N, ADJ, TX>(g, b, t, false, bd, false)) {
        tile_step<N, ADJ, TX, true, false>(&tm_lp, g, b, ac, an, t, mrev, nullptr, 0.0f, bd, Save2{-1, -1, nullptr}, inj, sm,
                                    &bar, err);
    } else {
        tile_step<N, ADJ, TX, false, false>(&tm_lp, g, b, ac, an, t, mrev, nullptr, 0.0f, bd, Save2{-1, -1, nullptr}, inj,
                                     sm, &bar, err);
    }
}

// Most tiles of a shot of the batch along z and x, for boxes [lo, hi].
struct Extent2 {
    int nz = 0, nx = 0;
    void add(int tx, const int lo[3], const int hi[3])
    {
        if (hi[0] < lo[0] || hi[1] < lo[1]) return;
        nz = std::max(nz, (hi[0] - (lo[0] & ~3)) / 32 + 1);
        nx = std::max(nx, (hi[1] - lo[1]) / tx + 1);
    }
};

}  // namespace

bool stencil2d_supported(const Grid &g)
{
    return g.ndim == 2 && (g.N == 2 || g.N == 4) && g.ntot < (1LL << 31) && tile_maps_available();
}

Step2 step2_tile(const Grid &g, int nshot)
{
    const long long tiles = (long long)((g.ne[0] + 31) / 32) * ((g.ne[1] + 31) / 32) * nshot;
    return Step2{tiles >= kMany};
}

bool make_maps2(Maps2 &m, const Grid &g, const Fields &f, int nshot, const Step2 &t, bool adjoint)
{
    const int rev = t.many ? 32 : 16, step = adjoint ? rev : kFwdTX;
    return make_tile_map(&m.p, g, f.p, nshot, 48, step + 4 * g.N - 2) &&
           make_tile_map(&m.vz, g, f.v[0], nshot, 48, rev + 2 * g.N - 1) &&
           make_tile_map(&m.vx, g, f.v[1], nshot, 40, rev + 4 * g.N - 2);
}

namespace {

template <int N, int BLOCKS>
void run_fwd(const LaunchCtx &lc, const Maps2 &mc, const Grid &g, const Batch &b, const Fields &c, const Fields &n, int step,
             const float *stf, float src_scale, const Bands &bd, const Save2 &save, const Gather2 &ga, unsigned *err)
{
    constexpr int TX = kFwdTX;
    Extent2 e;
    bool images = false;                      // a box holds mirrors of image rows that its tiles may not hold
    for (int s = 0; s < b.nshot; s++) {
        int lo[3], hi[3];
        box_bounds(g, b.h_box_src + 6 * s, step, lo, hi);
        e.add(TX, lo, hi);
        images = images || (g.freesurf && lo[0] > g.L[0] - N && lo[0] <= g.L[0] + N);
    }
    const int per = std::max(1, e.nz) * 8 * TX;
    const int ng = ga.it >= 0 ? (b.max_rec + per - 1) / per : 0;
    auto *kernel = save.amax ? k2_fwd<N, BLOCKS, true> : k2_fwd<N, BLOCKS, false>;
    for (int y0 = 0; y0 < e.nx + ng; y0 += kMaxRows)
        launch_pdl(lc, kernel, dim3(std::max(1, e.nz), std::min(kMaxRows, e.nx + ng - y0), b.nshot), 8 * TX, 0, mc.p, g, b,
                   c, n, step, stf, src_scale, bd, save, ga, ng, y0, err);
    // the few steps in which a deep source's box grows through the rows next to the surface; starting
    // every step's tiles at the image rows instead cost all launches 40 ns (201 x 201: 3.25 -> 3.29 us)
    if (images) launch_free_surface(lc, g, n.p, b.nshot, kFsMirrorP);
}

template <int N, int TX>
void run_rev(const LaunchCtx &lc, const Maps2 &mac, const Maps2 &mfc, const Grid &g, const Batch &b, const Fields &ac,
             const Fields &an, int mrev, int roles, const Fields &fc, const Fields &fn, int it, float *acc, int img_mode,
             const float *stf, float src_scale, const Bands &bd, bool restore, const Inject2 &ij, unsigned *err)
{
    Extent2 e;
    for (int s = 0; s < b.nshot; s++) {
        int lo[3], hi[3];
        if (roles & 1) {
            box_bounds(g, b.h_box_rec + 6 * s, mrev, lo, hi);
            e.add(TX, lo, hi);
        }
        if (!(roles & 2)) continue;
        box_bounds(g, b.h_box_src + 6 * s, std::min(it + 1, b.nt1 - 2), lo, hi);
        for (int a = 0; a < 2; a++) {
            lo[a] = std::max(lo[a], g.L[a] - N);
            hi[a] = std::min(hi[a], g.H[a] + N - 1);
        }
        e.add(TX, lo, hi);
    }
    for (int y0 = 0; y0 < e.nx; y0 += kMaxRows)
        launch_pdl(lc, k2_rev<N, TX>, dim3(e.nz, std::min(kMaxRows, e.nx - y0), b.nshot * (roles == 3 ? 2 : 1)), 8 * TX, 0,
                   mac.p, mfc.vz, mfc.vx, g, b, ac, an, mrev, roles, fc, fn, it, acc, img_mode, stf, src_scale, bd,
                   restore ? 1 : 0, ij, y0, err);
}

}  // namespace

void launch2_forward(const LaunchCtx &lc, const Step2 &t, const Maps2 &mc, const Grid &g, const Batch &b, Fields c,
                     Fields n, int step, const float *stf, float src_scale, const Bands &bd, Save2 save, Gather2 ga,
                     unsigned *err)
{
    if (g.N == 2 && !t.many) run_fwd<2, 4>(lc, mc, g, b, c, n, step, stf, src_scale, bd, save, ga, err);
    else if (g.N == 2) run_fwd<2, 6>(lc, mc, g, b, c, n, step, stf, src_scale, bd, save, ga, err);
    else if (!t.many) run_fwd<4, 4>(lc, mc, g, b, c, n, step, stf, src_scale, bd, save, ga, err);
    else run_fwd<4, 6>(lc, mc, g, b, c, n, step, stf, src_scale, bd, save, ga, err);
}

void launch2_reverse(const LaunchCtx &lc, const Step2 &t, const Maps2 &mac, const Maps2 &mfc, const Grid &g,
                     const Batch &b, Fields ac, Fields an, int mrev, int roles, Fields fc, Fields fn, int it,
                     float *acc, int img_mode, const float *stf, float src_scale, const Bands &bd, bool restore,
                     Inject2 ij, unsigned *err)
{
    if (g.N == 2 && !t.many)
        run_rev<2, 16>(lc, mac, mfc, g, b, ac, an, mrev, roles, fc, fn, it, acc, img_mode, stf, src_scale, bd, restore, ij, err);
    else if (g.N == 2)
        run_rev<2, 32>(lc, mac, mfc, g, b, ac, an, mrev, roles, fc, fn, it, acc, img_mode, stf, src_scale, bd, restore, ij, err);
    else if (!t.many)
        run_rev<4, 16>(lc, mac, mfc, g, b, ac, an, mrev, roles, fc, fn, it, acc, img_mode, stf, src_scale, bd, restore, ij, err);
    else
        run_rev<4, 32>(lc, mac, mfc, g, b, ac, an, mrev, roles, fc, fn, it, acc, img_mode, stf, src_scale, bd, restore, ij, err);
}

}  // namespace smi
