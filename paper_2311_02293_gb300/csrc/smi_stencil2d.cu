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
// 16.9 -> 3.7 us a step; 257 x 903 order 8 gradient, one shot, 16-bit
// boundaries, 69.5 -> 20.6 us a step pair; 301 x 1001, 40 shots, 315 -> 223.
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

__device__ __forceinline__ float4 ld4(const float *p) { return *reinterpret_cast<const float4 *>(p); }
__device__ __forceinline__ void st4(float *p, const float (&a)[4])
{
    *reinterpret_cast<float4 *>(p) = make_float4(a[0], a[1], a[2], a[3]);
}
__device__ __forceinline__ void window(float (&W)[12], const float *row)
{
#pragma unroll
    for (int k = 0; k < 3; k++) {
        const float4 a = ld4(row + 4 * k);
        W[4 * k] = a.x;
        W[4 * k + 1] = a.y;
        W[4 * k + 2] = a.z;
        W[4 * k + 3] = a.w;
    }
}
// Derivative along z of the quad in the middle of a 12-value window, p nodes
// to v nodes (UP) or back.
template <int N, bool UP> __device__ __forceinline__ void dz4(const Grid &g, const float (&W)[12], float (&D)[4])
{
#pragma unroll
    for (int r = 0; r < 4; r++) {
        float d = 0.0f;
#pragma unroll
        for (int l = 1; l <= N; l++)
            d += g.c[0][l - 1] * (UP ? W[4 + r + l] - W[4 + r - l + 1] : W[4 + r + l - 1] - W[4 + r - l]);
        D[r] = d;
    }
}
__device__ __forceinline__ void buoy4(const float (&r0)[4], const float (&r1)[4], float (&b)[4])
{
    // fast reciprocal-based division: a few ulp, far below the FP32 scheme error
#pragma unroll
    for (int r = 0; r < 4; r++) b[r] = __fdividef(2.0f, r0[r] + r1[r]);
}
// rho of the quad and of the quad one node up the axis (the last node's
// neighbour is itself: 2 / (rho + rho) = 1 / rho).
__device__ __forceinline__ void rho_z(const Grid &g, int oz, int k, float (&r0)[4], float (&r1)[4])
{
    put(r0, ld4(g.rho + k));
    const float up = oz + 4 < g.ne[0] ? g.rho[k + 4] : r0[3];
#pragma unroll
    for (int r = 0; r < 4; r++) {
        const float nx = r < 3 ? r0[r + 1] : up;
        r1[r] = oz + r + 1 < g.ne[0] ? nx : r0[r];
    }
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
__device__ __forceinline__ void add_source(const Batch &b, const SrcBox &sb, int s, int oz, int ox, float amp, float (&p)[4])
{
    const int t1 = ox - sb.f1;
    if (t1 < 0 || t1 >= sb.n1 || oz + 3 < sb.f0 || oz >= sb.f0 + sb.n0) return;
    const Stencil &st = b.src[s];
#pragma unroll
    for (int r = 0; r < 4; r++) {
        const int t0 = oz + r - sb.f0;
        if (t0 >= 0 && t0 < sb.n0) p[r] += amp * st.w[0][t0] * st.w[1][t1] * st.w[2][0];
    }
}

// Boundary regions of axis A at node (z, x): side 0 / 1, or -1.
template <int A> __device__ __forceinline__ int band_side(const Bands &bd, int z, int x)
{
#pragma unroll
    for (int sd = 0; sd < 2; sd++)
        if (in_range(z, bd.lo[A][sd][0], bd.hi[A][sd][0]) && in_range(x, bd.lo[A][sd][1], bd.hi[A][sd][1])) return sd;
    return -1;
}
template <int A> __device__ __forceinline__ long long band_off(const Bands &bd, int s, int it, int sd, int z, int x)
{
    const int w0 = bd.hi[A][sd][0] - bd.lo[A][sd][0] + 1;
    return ((long long)s * bd.nt + it) * bd.count + bd.off[A][sd] + (z - bd.lo[A][sd][0]) +
           (long long)w0 * (x - bd.lo[A][sd][1]);
}
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
// maps to 2^14 (FP16) or 1 (BF16).
template <int A>
__device__ __forceinline__ void band_store(const Bands &bd, const float (&scale)[4], int s, int it, int oz, int x,
                                           const float (&v)[4])
{
#pragma unroll
    for (int r = 0; r < 4; r++) {
        const int sd = band_side<A>(bd, oz + r, x);
        if (sd < 0) continue;
        const long long o = band_off<A>(bd, s, it, sd, oz + r, x);
        if (bd.prec == SMI_PREC_F32) {
            static_cast<float *>(bd.data)[o] = v[r];
        } else {
            const float sc = sd == 0 ? scale[2 * A] : scale[2 * A + 1];
            const float y = sc > 0.0f ? v[r] / sc : 0.0f;
            if (bd.prec == SMI_PREC_F16) static_cast<__half *>(bd.data)[o] = __float2half_rn(y);
            else static_cast<__nv_bfloat16 *>(bd.data)[o] = __float2bfloat16_rn(y);
        }
    }
}
// One velocity quad of axis A from the tile's pressure: v -= dt b D at the
// nodes of the box, memory variable m of the v grid, and the operand R that
// the pressure update differentiates (forward: v; adjoint: v + e).
// D: derivative of the axis; B, Av: the quad's CPML coefficients.
template <int MODE>
__device__ __forceinline__ void vel_quad(float dt, const float (&D)[4], const float (&b)[4], const bool (&in)[4],
                                         bool slab, const float (&B)[4], const float (&Av)[4], float (&m)[4],
                                         float (&v)[4], float (&R)[4])
{
#pragma unroll
    for (int r = 0; r < 4; r++) {
        float d = D[r];
        if (MODE == FWD && slab && in[r]) {
            m[r] = slab_recur(B[r], m[r], Av[r], d);
            d += m[r];
        }
        if (in[r]) v[r] -= dt * b[r] * d;
        R[r] = v[r];
        if (MODE == ADJ && slab) {
            if (in[r]) m[r] = slab_recur(B[r], m[r], Av[r], v[r]);
            R[r] += m[r];
        }
    }
}

// Forward or adjoint step of one tile.  sm: the block's shared tiles.
template <int N, int MODE, int TX>
__device__ __forceinline__ void tile_step(const CUtensorMap *tm_p, const Grid &g, const Batch &b, const Fields &c,
                                          const Fields &n, const Tile &t, int step, const float *stf, float src_scale,
                                          const Bands &bd, const Save2 &save, float *sm, uint64_t *bar,
                                          unsigned *smax, unsigned *err)
{
    using La = Lay<N, TX>;
    constexpr int HX = 2 * N - 1, NT = 8 * TX;
    float *sp = sm, *svz = sm + La::P, *svx = svz + La::VZ;
    const int tid = threadIdx.x, tzi = tid & 7, txi = tid >> 3;
    const int s = t.s, z0 = t.z0, x0 = t.x0;
    const int oz = z0 + 4 * tzi, ox = x0 + txi, k = oz + g.px * ox;
    const bool own = oz < g.ne[0] && ox < g.ne[1];
    const long long sh = (long long)s * g.ntot;
    const long long so0 = (long long)s * g.slab_n[0], so1 = (long long)s * g.slab_n[1];
    const float dt = g.dt;

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
    const bool ein = extra && ez >= 0 && ez < g.ne[0] && ex >= 0 && ex < g.ne[1];
    const int ke = ez + g.px * ex;

    // ---- what no earlier step writes: model, coefficients, source stencil ----
    float bz[4], bx[4], be[4], Kv[4];
    {
        float r0[4] = {1.0f, 1.0f, 1.0f, 1.0f}, r1[4] = {1.0f, 1.0f, 1.0f, 1.0f};
        if (own) rho_z(g, oz, k, r0, r1);
        buoy4(r0, r1, bz);
        if (own && ox + 1 < g.ne[1]) put(r1, ld4(g.rho + k + g.px));
        else for (int r = 0; r < 4; r++) r1[r] = r0[r];
        buoy4(r0, r1, bx);
        for (int r = 0; r < 4; r++) Kv[r] = 0.0f;
        if (own) put(Kv, ld4(g.K + k));
        if (ein) {
            if (exz) {
                rho_z(g, ez, ke, r0, r1);
            } else {
                put(r0, ld4(g.rho + ke));
                if (ex + 1 < g.ne[1]) put(r1, ld4(g.rho + ke + g.px));
                else for (int r = 0; r < 4; r++) r1[r] = r0[r];
            }
        }
        buoy4(r0, r1, be);
    }
    const int zq = own ? zslab_quad(g, oz) : -1, xq = own ? slab_row(g, 1, ox) : -1;
    const int eq = ein ? (exz ? zslab_quad(g, ez) : slab_row(g, 1, ex)) : -1;
    const long long zo = so0 + zq + (long long)g.zp * ox, xo = so1 + (long long)g.px * xq + oz;
    const long long eo = exz ? so0 + eq + (long long)g.zp * ex : so1 + (long long)g.px * eq + ez;
    SrcBox sb{0, 0, 0, 0};
    float amp = 0.0f;
    if (MODE == FWD && stf) {
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
    float vz[4] = {}, vx[4] = {}, ve[4] = {}, mz[4] = {}, mx[4] = {}, me[4] = {}, pz[4] = {}, px[4] = {};
    if (own) {
        put(vz, ld4(c.v[0] + sh + k));
        put(vx, ld4(c.v[1] + sh + k));
    }
    if (ein) put(ve, ld4((exz ? c.v[0] : c.v[1]) + sh + ke));
    if (zq >= 0) {
        put(mz, ld4(c.psip[0] + zo));
        put(pz, ld4(c.psiv[0] + zo));
    }
    if (xq >= 0) {
        put(mx, ld4(c.psip[1] + xo));
        put(px, ld4(c.psiv[1] + xo));
    }
    if (eq >= 0) put(me, ld4((exz ? c.psip[0] : c.psip[1]) + eo));

    const bool first = blockIdx.x == 0 && blockIdx.y == 0;      // writes the shot's scales
    if (MODE == FWD && save.sample >= 0 && (first || band_tile<TX>(bd, z0, x0))) {
        float scale[4] = {0.0f, 0.0f, 0.0f, 0.0f};
        if (bd.prec != SMI_PREC_F32) {
#pragma unroll
            for (int q = 0; q < 4; q++) {
                scale[q] = __uint_as_float(save.amax[((long long)save.sample * b.nshot + s) * 6 + q]) /
                           (bd.prec == SMI_PREC_F16 ? 16384.0f : 1.0f);
                if (first && tid == q) bd.scale[((long long)s * bd.nt + save.sample) * 6 + q] = scale[q];
            }
        }
        if (own) {
            band_store<0>(bd, scale, s, save.sample, oz, ox, vz);
            band_store<1>(bd, scale, s, save.sample, oz, ox, vx);
        }
    }

    if (!mbar_wait(bar, 0)) {                 // every thread gives up alike after the same number of polls
        if (tid == 0) atomicOr(err, 1u);
        mbar_wait(bar, 0);
    }

    // ---- velocities: own quads, then the halo's ----
    const bool inx = in_range(ox, t.lo[1], t.hi[1]);
    bool in[4];
#pragma unroll
    for (int r = 0; r < 4; r++) in[r] = inx && in_range(oz + r, t.lo[0], t.hi[0]);
    auto z_deriv = [&](int qz, int qx, float (&D)[4]) {
        float W[12];
        window(W, sp + (qx - x0 + HX) * La::PW + (qz - z0) + 4);
        if (MODE == ADJ && (qz - 4 < g.zlo || qz + 7 >= g.zhi) && qx >= 0 && qx < g.ne[1]) {
#pragma unroll
            for (int q = 0; q < 3; q++) {
                const int e = zslab_quad(g, qz - 4 + 4 * q);
                if (e < 0) continue;
                float a[4];
                put(a, ld4(c.psiv[0] + so0 + e + (long long)g.zp * qx));
#pragma unroll
                for (int r = 0; r < 4; r++) W[4 * q + r] += a[r];
            }
        }
        dz4<N, true>(g, W, D);
    };
    auto x_deriv = [&](int qz, int qx, float (&D)[4]) {
#pragma unroll
        for (int r = 0; r < 4; r++) D[r] = 0.0f;
        const bool near = MODE == ADJ && (qx - N + 1 < g.nb || qx + N >= g.ne[1] - g.nb - 1);
#pragma unroll
        for (int l = 1; l <= N; l++) {
            float a[4], d[4];
            const float *row = sp + (qx - x0 + HX) * La::PW + (qz - z0) + 8;
            put(a, ld4(row + l * La::PW));
            put(d, ld4(row - (l - 1) * La::PW));
            if (near && qz < g.ne[0]) {
                const int ja = slab_row(g, 1, qx + l), jd = slab_row(g, 1, qx - l + 1);
                float e[4];
                if (ja >= 0) {
                    put(e, ld4(c.psiv[1] + so1 + (long long)g.px * ja + qz));
#pragma unroll
                    for (int r = 0; r < 4; r++) a[r] += e[r];
                }
                if (jd >= 0) {
                    put(e, ld4(c.psiv[1] + so1 + (long long)g.px * jd + qz));
#pragma unroll
                    for (int r = 0; r < 4; r++) d[r] += e[r];
                }
            }
#pragma unroll
            for (int r = 0; r < 4; r++) D[r] += g.c[1][l - 1] * (a[r] - d[r]);
        }
    };
    {
        float D[4], R[4], B[4] = {}, Av[4] = {};
        z_deriv(oz, ox, D);
        if (zq >= 0) {
            put(B, ld4(g.cvb[0] + oz));
            put(Av, ld4(g.cva[0] + oz));
        }
        vel_quad<MODE>(dt, D, bz, in, zq >= 0, B, Av, mz, vz, R);
        st4(svz + txi * La::VW + 4 * tzi + 4, R);
        x_deriv(oz, ox, D);
        if (xq >= 0) {
            const float bb = g.cvb[1][ox], aa = g.cva[1][ox];
#pragma unroll
            for (int r = 0; r < 4; r++) {
                B[r] = bb;
                Av[r] = aa;
            }
        }
        vel_quad<MODE>(dt, D, bx, in, xq >= 0, B, Av, mx, vx, R);
        st4(svx + (txi + N) * 32 + 4 * tzi, R);
    }
    if (extra) {
        float D[4], R[4], B[4] = {}, Av[4] = {};
        bool ie[4];
        const bool iex = in_range(ex, t.lo[1], t.hi[1]);
#pragma unroll
        for (int r = 0; r < 4; r++) ie[r] = iex && in_range(ez + r, t.lo[0], t.hi[0]);
        if (exz) {
            z_deriv(ez, ex, D);
            if (eq >= 0) {
                put(B, ld4(g.cvb[0] + ez));
                put(Av, ld4(g.cva[0] + ez));
            }
        } else {
            x_deriv(ez, ex, D);
            if (eq >= 0) {
#pragma unroll
                for (int r = 0; r < 4; r++) {
                    B[r] = g.cvb[1][ex];
                    Av[r] = g.cva[1][ex];
                }
            }
        }
        vel_quad<MODE>(dt, D, be, ie, eq >= 0, B, Av, me, ve, R);
        if (exz) st4(svz + (ex - x0) * La::VW + (ez - z0 + 4), R);
        else st4(svx + (ex - x0 + N) * 32 + (ez - z0), R);
    }
    __syncthreads();
    if (g.freesurf && z0 - 4 < g.L[0]) {
        // free surface (image method): half node L-1-j mirrors L+j; the adjoint folds it there.  The box
        // starts at L-N or below the image rows, so a tile that holds an image row holds its mirror; the
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
        if (oz < L + N) put(vz, ld4(svz + txi * La::VW + 4 * tzi + 4));
    }

    // ---- pressure ----
    float pv[4], div[4];
    put(pv, ld4(sp + (txi + HX) * La::PW + 4 * tzi + 8));
    {
        float W[12], D[4];
        window(W, svz + txi * La::VW + 4 * tzi);
        dz4<N, false>(g, W, D);
        if (MODE == FWD && zq >= 0) {
            float B[4], A[4];
            put(B, ld4(g.cpb[0] + oz));
            put(A, ld4(g.cpa[0] + oz));
#pragma unroll
            for (int r = 0; r < 4; r++)
                if (in[r]) {
                    pz[r] = slab_recur(B[r], pz[r], A[r], D[r]);
                    D[r] += pz[r];
                }
        }
#pragma unroll
        for (int r = 0; r < 4; r++) {
            div[r] = D[r];
            D[r] = 0.0f;
        }
#pragma unroll
        for (int l = 1; l <= N; l++) {
            float a[4], d[4];
            put(a, ld4(svx + (txi + N + l - 1) * 32 + 4 * tzi));
            put(d, ld4(svx + (txi + N - l) * 32 + 4 * tzi));
#pragma unroll
            for (int r = 0; r < 4; r++) D[r] += g.c[1][l - 1] * (a[r] - d[r]);
        }
        if (MODE == FWD && xq >= 0) {
            const float B = g.cpb[1][ox], A = g.cpa[1][ox];
#pragma unroll
            for (int r = 0; r < 4; r++)
                if (in[r]) {
                    px[r] = slab_recur(B, px[r], A, D[r]);
                    D[r] += px[r];
                }
        }
#pragma unroll
        for (int r = 0; r < 4; r++) {
            div[r] += D[r];
            if (in[r]) pv[r] -= dt * Kv[r] * div[r];
        }
        if (MODE == ADJ && zq >= 0) {
            float B[4], A[4];
            put(B, ld4(g.cpb[0] + oz));
            put(A, ld4(g.cpa[0] + oz));
#pragma unroll
            for (int r = 0; r < 4; r++)
                if (in[r]) pz[r] = slab_recur(B[r], pz[r], A[r], pv[r]);
        }
        if (MODE == ADJ && xq >= 0) {
            const float B = g.cpb[1][ox], A = g.cpa[1][ox];
#pragma unroll
            for (int r = 0; r < 4; r++)
                if (in[r]) px[r] = slab_recur(B, px[r], A, pv[r]);
        }
    }
    if (MODE == FWD && stf) add_source(b, sb, s, oz, ox, amp, pv);
    if (MODE == FWD && g.freesurf && z0 <= g.L[0] + N) {
        // p = 0 on the surface row L, -p mirrored above it (the own pressures of the tile's centre)
        st4(sp + (txi + HX) * La::PW + 4 * tzi + 8, pv);
        __syncthreads();
        const int L = g.L[0];
#pragma unroll
        for (int r = 0; r < 4; r++) {
            const int z = oz + r, zm = 2 * L - z - z0;
            if (z == L) pv[r] = 0.0f;
            else if (z < L && z >= L - N && zm < 32) pv[r] = -sp[(txi + HX) * La::PW + zm + 8];
        }
    }
    if (own) {
        st4(n.v[0] + sh + k, vz);
        st4(n.v[1] + sh + k, vx);
        st4(n.p + sh + k, pv);
        if (zq >= 0) {
            st4(n.psip[0] + zo, mz);
            st4(n.psiv[0] + zo, pz);
        }
        if (xq >= 0) {
            st4(n.psip[1] + xo, mx);
            st4(n.psiv[1] + xo, px);
        }
    }
    if (MODE == FWD && save.next >= 0 && band_tile<TX>(bd, z0, x0)) {
        // largest magnitude per (axis, side) of the velocities the next sample stores
        if (tid < 4) smax[tid] = 0u;
        __syncthreads();
        if (own) {
#pragma unroll
            for (int r = 0; r < 4; r++) {
                const int s0 = band_side<0>(bd, oz + r, ox), s1 = band_side<1>(bd, oz + r, ox);
                if (s0 >= 0 && vz[r] != 0.0f) atomicMax(smax + s0, __float_as_uint(fabsf(vz[r])));
                if (s1 >= 0 && vx[r] != 0.0f) atomicMax(smax + 2 + s1, __float_as_uint(fabsf(vx[r])));
            }
        }
        __syncthreads();
        if (tid < 4 && smax[tid]) atomicMax(save.amax + ((long long)save.next * b.nshot + s) * 6 + tid, smax[tid]);
    }
}

template <int N, int TX>
__global__ void __launch_bounds__(8 * TX, TX == 32 ? 3 : 6)
k2_fwd(const __grid_constant__ CUtensorMap tm_p, Grid g, Batch b, Fields c, Fields n, int step, const float *stf,
       float src_scale, Bands bd, Save2 save, Gather2 ga, int nxt, unsigned *err)
{
    __shared__ __align__(128) float sm[Lay<N, TX>::FA];
    __shared__ __align__(8) uint64_t bar;
    __shared__ unsigned smax[4];
    Tile t;
    t.s = blockIdx.z;
    if ((int)blockIdx.y >= nxt) {              // receivers: samples of the pressure before the step
        pdl_wait();
        pdl_trigger();
        const int nr = b.rec_off[t.s + 1] - b.rec_off[t.s];
        const int r = ((blockIdx.y - nxt) * gridDim.x + blockIdx.x) * (8 * TX) + threadIdx.x;
        if (r >= nr) return;
        const Stencil &st = b.rec[b.rec_off[t.s] + r];
        const float *ps = c.p + t.s * g.ntot;
        float sum = 0.0f;
        for (int a1 = 0; a1 < st.cnt[1]; a1++)
            for (int a0 = 0; a0 < st.cnt[0]; a0++)
                sum += st.w[0][a0] * st.w[1][a1] * st.w[2][0] * ps[st.first[0] + a0 + g.px * (st.first[1] + a1)];
        ga.seis[ga.off[t.s] + (long long)ga.it * nr + r] = sum;
        return;
    }
    box_at(b.tab_src, b.nt1, t.s, step, t.lo, t.hi);
    t.z0 = (t.lo[0] & ~3) + 32 * blockIdx.x;
    t.x0 = t.lo[1] + TX * blockIdx.y;
    if (t.z0 > t.hi[0] || t.x0 > t.hi[1]) {
        if (blockIdx.x + blockIdx.y + blockIdx.z == 0) pdl_wait();   // one block of a launch always waits
        return;
    }
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        mbar_fence_init();
    }
    __syncthreads();
    tile_step<N, FWD, TX>(&tm_p, g, b, c, n, t, step, stf, src_scale, bd, save, sm, &bar, smax, err);
}

// Reconstruction of one tile.  Own nodes: the physical domain and the
// boundary bands inside the box of step it + 1 (so that nodes which left the
// box are written as zeros into both sets of arrays).
template <int N, int TX>
__device__ __forceinline__ void tile_rec(const CUtensorMap *tm_vz, const CUtensorMap *tm_vx, const Grid &g,
                                         const Batch &b, const Fields &c, const Fields &n, const Tile &t, int it,
                                         const float *lp, float *acc, int img_mode, const float *stf, float src_scale,
                                         const Bands &bd, bool restore, float *sm, uint64_t *bar, unsigned *err)
{
    using La = Lay<N, TX>;
    constexpr int HX = 2 * N - 1;
    float *tz = sm, *tx = sm + La::RZ, *spn = tx + La::RX;
    const int tid = threadIdx.x, tzi = tid & 7, txi = tid >> 3;
    const int s = t.s, z0 = t.z0, x0 = t.x0;
    const int oz = z0 + 4 * tzi, ox = x0 + txi, k = oz + g.px * ox;
    const bool own = oz < g.ne[0] && ox < g.ne[1];
    const long long sh = (long long)s * g.ntot;
    const float dt = g.dt;
    if (tid == 0) {
        mbar_expect(bar, (unsigned)(La::RZB + La::RXB) * 4u);
        tma4(tz, tm_vz, z0 - 8, x0 - N + 1, 0, s, bar);
        tma4(tx, tm_vx, z0 - 4, x0 - HX, 0, s, bar);
    }
    // update region (box of the step within the physical domain), previous box
    int plo[3], phi[3], lo[2], hi[2];
    box_at(b.tab_src, b.nt1, s, it - 1, plo, phi);
    {
        int bl[3], bh[3];
        box_at(b.tab_src, b.nt1, s, it, bl, bh);
#pragma unroll
        for (int a = 0; a < 2; a++) {
            lo[a] = max(bl[a], g.L[a]);
            hi[a] = min(bh[a], g.H[a]);
        }
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
    const bool ein = extra && ez >= 0 && ez < g.ne[0] && ex >= 0 && ex < g.ne[1];
    const int ke = ez + g.px * ex;

    float bz[4], bx[4], Kv[4] = {}, Ke[4] = {}, pv[4] = {}, pe[4] = {}, lpv[4] = {};
    {
        float r0[4] = {1.0f, 1.0f, 1.0f, 1.0f}, r1[4] = {1.0f, 1.0f, 1.0f, 1.0f};
        if (own) rho_z(g, oz, k, r0, r1);
        buoy4(r0, r1, bz);
        if (own && ox + 1 < g.ne[1]) put(r1, ld4(g.rho + k + g.px));
        else for (int r = 0; r < 4; r++) r1[r] = r0[r];
        buoy4(r0, r1, bx);
    }
    if (own) {
        put(Kv, ld4(g.K + k));
        put(pv, ld4(c.p + sh + k));
        put(lpv, ld4(lp + sh + k));
    }
    if (ein) {
        put(Ke, ld4(g.K + ke));
        put(pe, ld4(c.p + sh + ke));
    }
    const SrcBox sb = src_box(b, s);
    const float amp = -src_scale * stf[it];
    // image / gradient accumulator of the quad: one 16-byte access where it is whole and aligned
    bool in[4];
    const bool inx = in_range(ox, lo[1], hi[1]);
#pragma unroll
    for (int r = 0; r < 4; r++) in[r] = inx && in_range(oz + r, lo[0], hi[0]);
    const long long ka = (long long)s * g.nphys + (oz - g.L[0]) + (long long)(g.H[0] - g.L[0] + 1) * (ox - g.L[1]);
    const bool acc4 = in[0] && in[3] && (ka & 3) == 0;
    float av[4] = {};
    if (acc4) {
        put(av, ld4(acc + ka));
    } else {
#pragma unroll
        for (int r = 0; r < 4; r++)
            if (in[r]) av[r] = acc[ka + r];
    }
    const bool bands = band_tile<TX>(bd, z0, x0);
    float scale[4] = {1.0f, 1.0f, 1.0f, 1.0f};
    if (restore && bands && bd.prec != SMI_PREC_F32) {
#pragma unroll
        for (int q = 0; q < 4; q++) scale[q] = bd.scale[((long long)s * bd.nt + it) * 6 + q];
    }
    if (!mbar_wait(bar, 0)) {
        if (tid == 0) atomicOr(err, 1u);
        mbar_wait(bar, 0);
    }

    // ---- pressures: p + dt kappa div v - source, zero outside the previous box ----
    auto press = [&](int qz, int qx, const float (&K4)[4], float (&p)[4], float (&dv)[4]) {
        float W[12], D[4];
        window(W, tz + (qx - x0 + N - 1) * La::PW + (qz - z0) + 4);
        dz4<N, false>(g, W, dv);
#pragma unroll
        for (int r = 0; r < 4; r++) D[r] = 0.0f;
        const float *row = tx + (qx - x0 + HX) * La::VW + (qz - z0) + 4;
#pragma unroll
        for (int l = 1; l <= N; l++) {
            float a[4], d[4];
            put(a, ld4(row + (l - 1) * La::VW));
            put(d, ld4(row - l * La::VW));
#pragma unroll
            for (int r = 0; r < 4; r++) D[r] += g.c[1][l - 1] * (a[r] - d[r]);
        }
        float q[4];
#pragma unroll
        for (int r = 0; r < 4; r++) {
            dv[r] += D[r];
            q[r] = p[r] + dt * K4[r] * dv[r];
        }
        add_source(b, sb, s, qz, qx, amp, q);
        const bool ix = in_range(qx, lo[1], hi[1]), kx = in_range(qx, plo[1], phi[1]);
#pragma unroll
        for (int r = 0; r < 4; r++) {
            if (!(ix && in_range(qz + r, lo[0], hi[0]))) continue;
            p[r] = (kx && in_range(qz + r, plo[0], phi[0]) && !(g.freesurf && qz + r == g.L[0])) ? q[r] : 0.0f;
        }
    };
    {
        float dv[4], np[4];
#pragma unroll
        for (int r = 0; r < 4; r++) np[r] = pv[r];
        press(oz, ox, Kv, np, dv);
        st4(spn + (txi + N - 1) * La::VW + 4 * tzi + 4, np);
        if (own) st4(n.p + sh + k, np);
#pragma unroll
        for (int r = 0; r < 4; r++) av[r] += lpv[r] * (img_mode == 0 ? dv[r] : pv[r]);
        if (acc4) {
            st4(acc + ka, av);
        } else {
#pragma unroll
            for (int r = 0; r < 4; r++)
                if (in[r]) acc[ka + r] = av[r];
        }
        if (img_mode == 2) {                   // illumination
#pragma unroll
            for (int r = 0; r < 4; r++)
                if (in[r]) acc[(long long)b.nshot * g.nphys + ka + r] += pv[r] * pv[r];
        }
    }
    if (extra) {
        float dv[4];
        press(ez, ex, Ke, pe, dv);
        st4(spn + (ex - x0 + N - 1) * La::VW + (ez - z0) + 4, pe);
    }
    float vz[4] = {}, vx[4] = {};
    put(vz, ld4(tz + (txi + N - 1) * La::PW + 4 * tzi + 8));
    put(vx, ld4(tx + (txi + HX) * La::VW + 4 * tzi + 4));
    __syncthreads();

    // ---- velocities: v_a + dt b_a D_a p on L_a+N-1 .. H_a-N, the bands from the store ----
    {
        float W[12], D[4], X[4] = {};
        window(W, spn + (txi + N - 1) * La::VW + 4 * tzi);
        dz4<N, true>(g, W, D);
#pragma unroll
        for (int l = 1; l <= N; l++) {
            float a[4], d[4];
            put(a, ld4(spn + (txi + N - 1 + l) * La::VW + 4 * tzi + 4));
            put(d, ld4(spn + (txi + N - l) * La::VW + 4 * tzi + 4));
#pragma unroll
            for (int r = 0; r < 4; r++) X[r] += g.c[1][l - 1] * (a[r] - d[r]);
        }
        const bool kx = in_range(ox, plo[1], phi[1]), rx = in_range(ox, g.L[1] + N - 1, g.H[1] - N);
#pragma unroll
        for (int r = 0; r < 4; r++) {
            const int z = oz + r;
            const bool keep = kx && in_range(z, plo[0], phi[0]);
            if (in[r] && in_range(z, g.L[0] + N - 1, g.H[0] - N)) vz[r] = keep ? vz[r] + dt * bz[r] * D[r] : 0.0f;
            if (in[r] && rx) vx[r] = keep ? vx[r] + dt * bx[r] * X[r] : 0.0f;
        }
        if (restore && bands) {
#pragma unroll
            for (int r = 0; r < 4; r++) {
                const int s0 = band_side<0>(bd, oz + r, ox), s1 = band_side<1>(bd, oz + r, ox);
                const bool keep = kx && in_range(oz + r, plo[0], phi[0]);      // zero (and not stored) outside
                if (s0 >= 0)
                    vz[r] = keep ? band_load(bd, band_off<0>(bd, s, it, s0, oz + r, ox), s0 ? scale[1] : scale[0]) : 0.0f;
                if (s1 >= 0)
                    vx[r] = keep ? band_load(bd, band_off<1>(bd, s, it, s1, oz + r, ox), s1 ? scale[3] : scale[2]) : 0.0f;
            }
        }
        if (own) {
            st4(n.v[0] + sh + k, vz);
            st4(n.v[1] + sh + k, vx);
        }
    }
}

// roles 1: adjoint, 2: reconstruction (blockIdx.z = shot), 3: both
// (blockIdx.z = 2 shot + role, 0 adjoint, 1 reconstruction).
template <int N, int TX>
__global__ void __launch_bounds__(8 * TX, TX == 32 ? 3 : 6)
k2_rev(const __grid_constant__ CUtensorMap tm_lp, const __grid_constant__ CUtensorMap tm_vz,
       const __grid_constant__ CUtensorMap tm_vx, Grid g, Batch b, Fields ac, Fields an, int mrev, int roles, Fields fc,
       Fields fn, int it, float *acc, int img_mode, const float *stf, float src_scale, Bands bd, int restore,
       unsigned *err)
{
    __shared__ __align__(128) float sm[Lay<N, TX>::MAXF];
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
    t.x0 = t.lo[1] + TX * blockIdx.y;
    if (t.z0 > t.hi[0] || t.x0 > t.hi[1]) {
        if (blockIdx.x + blockIdx.y + blockIdx.z == 0) pdl_wait();
        return;
    }
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        mbar_fence_init();
    }
    __syncthreads();
    pdl_wait();
    pdl_trigger();
    if (role)
        tile_rec<N, TX>(&tm_vz, &tm_vx, g, b, fc, fn, t, it, ac.p, acc, img_mode, stf, src_scale, bd, restore != 0, sm,
                        &bar, err);
    else
        tile_step<N, ADJ, TX>(&tm_lp, g, b, ac, an, t, mrev, nullptr, 0.0f, bd, Save2{-1, -1, nullptr}, sm, &bar,
                              nullptr, err);
}

// Most tiles of a shot of the batch along z and x, for boxes [lo, hi] clipped
// by clip_lo / clip_hi.
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

// Narrow tiles when the wide ones would not give every SM two blocks: the
// step is then bound by latency, and more, smaller blocks shorten it.
Step2 step2_tile(const Grid &g, int nshot)
{
    const long long tiles = (long long)((g.ne[0] + 31) / 32) * ((g.ne[1] + 31) / 32) * nshot;
    return Step2{tiles < 2 * 152 ? 16 : 32};
}

bool make_maps2(Maps2 &m, const Grid &g, const Fields &f, int nshot, const Step2 &t)
{
    const int pr = t.tx + 4 * g.N - 2, xr = t.tx + 2 * g.N - 1;
    return make_tile_map(&m.p, g, f.p, nshot, 48, pr) && make_tile_map(&m.vz, g, f.v[0], nshot, 48, xr) &&
           make_tile_map(&m.vx, g, f.v[1], nshot, 40, pr);
}

namespace {

template <int N, int TX>
void run_fwd(const LaunchCtx &lc, const Maps2 &mc, const Grid &g, const Batch &b, const Fields &c, const Fields &n, int step,
             const float *stf, float src_scale, const Bands &bd, const Save2 &save, const Gather2 &ga, unsigned *err)
{
    Extent2 e;
    for (int s = 0; s < b.nshot; s++) {
        int lo[3], hi[3];
        box_bounds(g, b.h_box_src + 6 * s, step, lo, hi);
        e.add(TX, lo, hi);
    }
    const int per = std::max(1, e.nz) * 8 * TX;
    const int ng = ga.it >= 0 ? (b.max_rec + per - 1) / per : 0;
    if (e.nx + ng == 0) return;
    launch_pdl(lc, k2_fwd<N, TX>, dim3(std::max(1, e.nz), e.nx + ng, b.nshot), 8 * TX, 0, mc.p, g, b, c, n, step, stf,
               src_scale, bd, save, ga, e.nx, err);
}

template <int N, int TX>
void run_rev(const LaunchCtx &lc, const Maps2 &mac, const Maps2 &mfc, const Grid &g, const Batch &b, const Fields &ac,
             const Fields &an, int mrev, int roles, const Fields &fc, const Fields &fn, int it, float *acc, int img_mode,
             const float *stf, float src_scale, const Bands &bd, bool restore, unsigned *err)
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
    if (e.nx == 0) return;
    launch_pdl(lc, k2_rev<N, TX>, dim3(e.nz, e.nx, b.nshot * (roles == 3 ? 2 : 1)), 8 * TX, 0, mac.p, mfc.vz, mfc.vx, g, b, ac,
               an, mrev, roles, fc, fn, it, acc, img_mode, stf, src_scale, bd, restore ? 1 : 0, err);
}

}  // namespace

void launch2_forward(const LaunchCtx &lc, const Step2 &t, const Maps2 &mc, const Grid &g, const Batch &b, Fields c,
                     Fields n, int step, const float *stf, float src_scale, const Bands &bd, Save2 save, Gather2 ga,
                     unsigned *err)
{
    if (g.N == 2 && t.tx == 16) run_fwd<2, 16>(lc, mc, g, b, c, n, step, stf, src_scale, bd, save, ga, err);
    else if (g.N == 2) run_fwd<2, 32>(lc, mc, g, b, c, n, step, stf, src_scale, bd, save, ga, err);
    else if (t.tx == 16) run_fwd<4, 16>(lc, mc, g, b, c, n, step, stf, src_scale, bd, save, ga, err);
    else run_fwd<4, 32>(lc, mc, g, b, c, n, step, stf, src_scale, bd, save, ga, err);
}

void launch2_reverse(const LaunchCtx &lc, const Step2 &t, const Maps2 &mac, const Maps2 &mfc, const Grid &g,
                     const Batch &b, Fields ac, Fields an, int mrev, int roles, Fields fc, Fields fn, int it,
                     float *acc, int img_mode, const float *stf, float src_scale, const Bands &bd, bool restore,
                     unsigned *err)
{
    if (g.N == 2 && t.tx == 16)
        run_rev<2, 16>(lc, mac, mfc, g, b, ac, an, mrev, roles, fc, fn, it, acc, img_mode, stf, src_scale, bd, restore, err);
    else if (g.N == 2)
        run_rev<2, 32>(lc, mac, mfc, g, b, ac, an, mrev, roles, fc, fn, it, acc, img_mode, stf, src_scale, bd, restore, err);
    else if (t.tx == 16)
        run_rev<4, 16>(lc, mac, mfc, g, b, ac, an, mrev, roles, fc, fn, it, acc, img_mode, stf, src_scale, bd, restore, err);
    else
        run_rev<4, 32>(lc, mac, mfc, g, b, ac, an, mrev, roles, fc, fn, it, acc, img_mode, stf, src_scale, bd, restore, err);
}

}  // namespace smi
