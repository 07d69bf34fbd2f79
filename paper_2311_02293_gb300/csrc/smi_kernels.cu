// smi_kernels.cu -- CUDA kernels of libsmi (sm_103a): staggered-grid
// velocity/pressure updates with slab-only CPML, source injection, receiver
// gather, boundary-band save/restore, residual/misfit, the exact discrete
// adjoint in "same solver" form, source-field reconstruction fused with
// imaging/gradient accumulation, and the device-side computing box.
//
// Every stencil kernel is bounded by the computing box of its shot (Sec.
// 4.1), computed on the device from the step counter; threads stride over
// the box's points.  Stencil reads outside the extended grid are zero.
#include <cuda_runtime.h>

#include <algorithm>
#include <cuda_fp16.h>
#include <cuda_bf16.h>

#include "smi_internal.h"
#include "smi_box.h"
#include "smi_band.h"
#include "smi_pdl.h"
#include "smi_slab.h"

namespace smi {

namespace {

constexpr int kThreads = 256;
constexpr int kMaxBlocksX = 152 * 16;

__device__ __forceinline__ long long gidx(const Grid &g, int i1, int i2, int i3)
{
    return (long long)i1 + (long long)g.px * ((long long)i2 + (long long)g.ne[1] * i3);
}

__device__ __forceinline__ long long gstride(const Grid &g, int a)
{
    return a == 0 ? 1LL : (a == 1 ? (long long)g.px : (long long)g.px * g.ne[1]);
}

// CPML slab membership along axis a: nodes 0..nb-1 and ne-nb-1..ne-1 (the
// latter covers the first v node of the high layer).
__device__ __forceinline__ bool in_slab(const Grid &g, int a, int j)
{
    return j < g.nb || j >= g.ne[a] - g.nb - 1;
}

// Index into the slab array of axis a (axis a compressed to S = 2nb+1).
__device__ __forceinline__ long long slab_index(const Grid &g, int a, int i1, int i2, int i3)
{
    if (a == 0) {
        int js = i1 < g.nb ? i1 : i1 - (g.ne[0] - 2 * g.nb - 1);
        return (long long)js + (long long)g.S * ((long long)i2 + (long long)g.ne[1] * i3);
    }
    if (a == 1) {
        int js = i2 < g.nb ? i2 : i2 - (g.ne[1] - 2 * g.nb - 1);
        return (long long)i1 + (long long)g.ne[0] * ((long long)js + (long long)g.S * i3);
    }
    int js = i3 < g.nb ? i3 : i3 - (g.ne[2] - 2 * g.nb - 1);
    return (long long)i1 + (long long)g.px * ((long long)i2 + (long long)g.ne[1] * js);
}

__device__ __forceinline__ float buoyancy(const Grid &g, int a, int ia, long long k, float rho0)
{
    // fast reciprocal-based division: a few ulp, far below the FP32 scheme error
    return (ia + 1 < g.ne[a]) ? __fdividef(2.0f, rho0 + g.rho[k + gstride(g, a)]) : __fdividef(1.0f, rho0);
}

struct BoxIter {
    int lo[3], hi[3];
    int w0, w1;
    long long vol;
    __device__ void set(const int l[3], const int h[3])
    {
        for (int a = 0; a < 3; a++) { lo[a] = l[a]; hi[a] = h[a]; }
        w0 = hi[0] - lo[0] + 1;
        w1 = hi[1] - lo[1] + 1;
        const int w2 = hi[2] - lo[2] + 1;
        vol = (w0 > 0 && w1 > 0 && w2 > 0) ? (long long)w0 * w1 * w2 : 0;
    }
    __device__ void at(long long q, int i[3]) const
    {
        if (vol < (1LL << 31)) {          // 32-bit division (uniform branch)
            const int qq = (int)q, r = qq / w0;
            i[0] = lo[0] + (qq - r * w0);
            i[1] = lo[1] + r % w1;
            i[2] = lo[2] + r / w1;
            return;
        }
        i[0] = lo[0] + (int)(q % w0);
        long long r = q / w0;
        i[1] = lo[1] + (int)(r % w1);
        i[2] = lo[2] + (int)(r / w1);
    }
};

__device__ __forceinline__ bool inside(const int i[3], const int lo[3], const int hi[3])
{
    return i[0] >= lo[0] && i[0] <= hi[0] && i[1] >= lo[1] && i[1] <= hi[1] && i[2] >= lo[2] &&
           i[2] <= hi[2];
}

// ---------------------------------------------------------------------------
// Forward velocity update (Sec. 2.1): v_a -= dt b_a (D_a p + psi_a), with the
// slab memory variable psi_a <- b psi_a + a D_a p updated first.
template <int NDIM, int N>
__global__ void __launch_bounds__(kThreads) k_fwd_v(Grid g, Batch b, Fields f, int it)
{
    const int s = blockIdx.y;
    int lo[3], hi[3];
    box_at(b.tab_src, b.nt1, s, it, lo, hi);
    BoxIter bi;
    bi.set(lo, hi);
    const float *p = f.p + s * g.ntot;
    for (long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x; q < bi.vol;
         q += (long long)gridDim.x * blockDim.x) {
        int i[3];
        bi.at(q, i);
        const long long k = gidx(g, i[0], i[1], i[2]);
        const float rho0 = g.rho[k];
#pragma unroll
        for (int a = 0; a < NDIM; a++) {
            const long long st = gstride(g, a);
            float D = 0.0f;
#pragma unroll
            for (int l = 1; l <= N; l++) {
                const float pp = (i[a] + l < g.ne[a]) ? p[k + l * st] : 0.0f;
                const float pm = (i[a] - l + 1 >= 0) ? p[k - (l - 1) * st] : 0.0f;
                D += g.c[a][l - 1] * (pp - pm);
            }
            if (in_slab(g, a, i[a])) {
                const long long si = s * g.slab_n[a] + slab_index(g, a, i[0], i[1], i[2]);
                const float psi = g.cvb[a][i[a]] * f.psip[a][si] + g.cva[a][i[a]] * D;
                f.psip[a][si] = psi;
                D += psi;
            }
            f.v[a][s * g.ntot + k] -= g.dt * buoyancy(g, a, i[a], k, rho0) * D;
        }
    }
}

// Forward pressure update: p -= dt kappa sum_a (D_a v_a + psi_a).
template <int NDIM, int N>
__global__ void __launch_bounds__(kThreads) k_fwd_p(Grid g, Batch b, Fields f, int it)
{
    const int s = blockIdx.y;
    int lo[3], hi[3];
    box_at(b.tab_src, b.nt1, s, it, lo, hi);
    BoxIter bi;
    bi.set(lo, hi);
    for (long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x; q < bi.vol;
         q += (long long)gridDim.x * blockDim.x) {
        int i[3];
        bi.at(q, i);
        const long long k = gidx(g, i[0], i[1], i[2]);
        float div = 0.0f;
#pragma unroll
        for (int a = 0; a < NDIM; a++) {
            const long long st = gstride(g, a);
            const float *v = f.v[a] + s * g.ntot;
            float D = 0.0f;
#pragma unroll
            for (int l = 1; l <= N; l++) {
                const float vp = (i[a] + l - 1 < g.ne[a]) ? v[k + (l - 1) * st] : 0.0f;
                const float vm = (i[a] - l >= 0) ? v[k - l * st] : 0.0f;
                D += g.c[a][l - 1] * (vp - vm);
            }
            if (in_slab(g, a, i[a])) {
                const long long si = s * g.slab_n[a] + slab_index(g, a, i[0], i[1], i[2]);
                const float psi = g.cpb[a][i[a]] * f.psiv[a][si] + g.cpa[a][i[a]] * D;
                f.psiv[a][si] = psi;
                D += psi;
            }
            div += D;
        }
        f.p[s * g.ntot + k] -= g.dt * g.K[k] * div;
    }
}

// ---------------------------------------------------------------------------
// Exact discrete adjoint in "same solver" form.  With lambda_p = kappa pbar
// and lambda_v = -b vbar (pbar, vbar the adjoints of p, v), the transpose of
// the forward step becomes, in reverse time:
//   V: lv_a -= dt b_a D_a[(1 + Ap_a) lp + Ap_a phi_a];   phi_a <- Bp_a (phi_a + lp)
//   P: lp   -= dt kappa sum_a D_a[(1 + Av_a) lv_a + Av_a chi_a];  chi_a <- Bv_a (chi_a + lv_a)
// (A, B the CPML a/b on the p grid (Ap, Bp) or v grid (Av, Bv)); in the
// interior this is the forward scheme itself (Sec. 2.2: the adjoint shares
// the forward solver).  phi lives on the p grid (stored in psiv), chi on
// the v grid (stored in psip).  The chi update of a reverse step is applied
// at the start of the next V kernel (it is pointwise), the phi update in the
// P kernel before lp changes.  m = reverse steps elapsed (box of the
// receivers, Sec. 4.1).
template <int NDIM, int N>
__global__ void __launch_bounds__(kThreads) k_adj_v(Grid g, Batch b, Fields f, int m)
{
    const int s = blockIdx.y;
    int lo[3], hi[3];
    box_at(b.tab_rec, b.nt1, s, m, lo, hi);
    BoxIter bi;
    bi.set(lo, hi);
    const float *lp = f.p + s * g.ntot;
    for (long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x; q < bi.vol;
         q += (long long)gridDim.x * blockDim.x) {
        int i[3];
        bi.at(q, i);
        const long long k = gidx(g, i[0], i[1], i[2]);
        const float rho0 = g.rho[k];
#pragma unroll
        for (int a = 0; a < NDIM; a++) {
            const long long st = gstride(g, a);
            float *lv = f.v[a] + s * g.ntot;
            if (in_slab(g, a, i[a])) {             // deferred chi update
                const long long si = s * g.slab_n[a] + slab_index(g, a, i[0], i[1], i[2]);
                f.psip[a][si] = g.cvb[a][i[a]] * (f.psip[a][si] + lv[k]);
            }
            float D = 0.0f;
#pragma unroll
            for (int l = 1; l <= N; l++) {
                float qv[2];
                const int off[2] = {l, 1 - l};
#pragma unroll
                for (int e = 0; e < 2; e++) {
                    int j[3] = {i[0], i[1], i[2]};
                    j[a] += off[e];
                    float val = 0.0f;
                    if (j[a] >= 0 && j[a] < g.ne[a]) {
                        const long long kk = k + off[e] * st;
                        val = lp[kk];
                        if (in_slab(g, a, j[a])) {
                            const float A = g.cpa[a][j[a]];
                            const long long sj = s * g.slab_n[a] + slab_index(g, a, j[0], j[1], j[2]);
                            val += A * (val + f.psiv[a][sj]);
                        }
                    }
                    qv[e] = val;
                }
                D += g.c[a][l - 1] * (qv[0] - qv[1]);
            }
            lv[k] -= g.dt * buoyancy(g, a, i[a], k, rho0) * D;
        }
    }
}

template <int NDIM, int N>
__global__ void __launch_bounds__(kThreads) k_adj_p(Grid g, Batch b, Fields f, int m)
{
    const int s = blockIdx.y;
    int lo[3], hi[3];
    box_at(b.tab_rec, b.nt1, s, m, lo, hi);
    BoxIter bi;
    bi.set(lo, hi);
    float *lp = f.p + s * g.ntot;
    for (long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x; q < bi.vol;
         q += (long long)gridDim.x * blockDim.x) {
        int i[3];
        bi.at(q, i);
        const long long k = gidx(g, i[0], i[1], i[2]);
        const float lpk = lp[k];
        float div = 0.0f;
#pragma unroll
        for (int a = 0; a < NDIM; a++) {
            const long long st = gstride(g, a);
            const float *lv = f.v[a] + s * g.ntot;
            if (in_slab(g, a, i[a])) {             // phi update with lp before this step
                const long long si = s * g.slab_n[a] + slab_index(g, a, i[0], i[1], i[2]);
                f.psiv[a][si] = g.cpb[a][i[a]] * (f.psiv[a][si] + lpk);
            }
            float D = 0.0f;
#pragma unroll
            for (int l = 1; l <= N; l++) {
                float rv[2];
                const int off[2] = {l - 1, -l};
#pragma unroll
                for (int e = 0; e < 2; e++) {
                    int j[3] = {i[0], i[1], i[2]};
                    j[a] += off[e];
                    float val = 0.0f;
                    if (j[a] >= 0 && j[a] < g.ne[a]) {
                        const long long kk = k + off[e] * st;
                        val = lv[kk];
                        if (in_slab(g, a, j[a])) {
                            const float A = g.cva[a][j[a]];
                            const long long sj = s * g.slab_n[a] + slab_index(g, a, j[0], j[1], j[2]);
                            val += A * (val + f.psip[a][sj]);
                        }
                    }
                    rv[e] = val;
                }
                D += g.c[a][l - 1] * (rv[0] - rv[1]);
            }
            div += D;
        }
        lp[k] = lpk - g.dt * g.K[k] * div;
    }
}

// ---------------------------------------------------------------------------
// Source-field reconstruction (Sec. 4.2, Algorithm 2 reverse loop) fused with
// the imaging / gradient accumulation, over the physical nodes of the
// forward box of step it:
//   acc += lp * div v^{it+1/2}  (gradient)   or  lp * p^{it+1}  (image)
//   p^{it} = p^{it+1} + dt kappa div v^{it+1/2} - dt stf[it] w / dV
// Nodes outside the box of step it-1 are set to zero (they were zero
// before step it).  lp is the adjoint pressure after the receivers of step
// it were injected.
template <int NDIM, int N>
__global__ void __launch_bounds__(kThreads)
k_recon_p(Grid g, Batch b, Fields f, const float *lpall, float *acc, int mode, const float *stf,
          int it, float src_scale)
{
    const int s = blockIdx.y;
    int lo[3], hi[3], plo[3], phi[3];
    box_at(b.tab_src, b.nt1, s, it, lo, hi);
    box_at(b.tab_src, b.nt1, s, it - 1, plo, phi);
    for (int a = 0; a < 3; a++) {
        lo[a] = max(lo[a], g.L[a]);
        hi[a] = min(hi[a], g.H[a]);
    }
    BoxIter bi;
    bi.set(lo, hi);
    float *p = f.p + s * g.ntot;
    const float *lp = lpall + s * g.ntot;
    const Stencil &sst = b.src[s];
    const float amp = src_scale * stf[it];
    for (long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x; q < bi.vol;
         q += (long long)gridDim.x * blockDim.x) {
        int i[3];
        bi.at(q, i);
        const long long k = gidx(g, i[0], i[1], i[2]);
        float dv = 0.0f;
#pragma unroll
        for (int a = 0; a < NDIM; a++) {
            const long long st = gstride(g, a);
            const float *v = f.v[a] + s * g.ntot;
            float D = 0.0f;
#pragma unroll
            for (int l = 1; l <= N; l++) D += g.c[a][l - 1] * (v[k + (l - 1) * st] - v[k - l * st]);
            dv += D;
        }
        const float pk = p[k];
        const long long kp = (long long)(i[0] - g.L[0]) +
                             (long long)(g.H[0] - g.L[0] + 1) *
                                 ((long long)(i[1] - g.L[1]) + (long long)(g.H[1] - g.L[1] + 1) * (i[2] - g.L[2]));
        acc[s * g.nphys + kp] += lp[k] * (mode == 0 ? dv : pk);
        if (mode == 2) acc[(long long)(b.nshot + s) * g.nphys + kp] += pk * pk;   // illumination
        float pn = pk + g.dt * g.K[k] * dv;
        bool in_src = true;
        float w = 1.0f;
#pragma unroll
        for (int a = 0; a < 3; a++) {
            const int t = i[a] - sst.first[a];
            in_src = in_src && t >= 0 && t < sst.cnt[a];
            if (in_src) w *= sst.w[a][t];
        }
        if (in_src) pn -= amp * w;
        if (!inside(i, plo, phi)) pn = 0.0f;
        p[k] = pn;
    }
}

// v_a^{it-1/2} = v_a^{it+1/2} + dt b_a D_a p^{it} on L_a+N-1 .. H_a-N along a
// (other axes over the physical nodes), inside the forward box of step it.
template <int NDIM, int N>
__global__ void __launch_bounds__(kThreads) k_recon_v(Grid g, Batch b, Fields f, int it)
{
    const int s = blockIdx.y;
    int lo[3], hi[3], plo[3], phi[3];
    box_at(b.tab_src, b.nt1, s, it, lo, hi);
    box_at(b.tab_src, b.nt1, s, it - 1, plo, phi);
    for (int a = 0; a < 3; a++) {
        lo[a] = max(lo[a], g.L[a]);
        hi[a] = min(hi[a], g.H[a]);
    }
    BoxIter bi;
    bi.set(lo, hi);
    const float *p = f.p + s * g.ntot;
    for (long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x; q < bi.vol;
         q += (long long)gridDim.x * blockDim.x) {
        int i[3];
        bi.at(q, i);
        const long long k = gidx(g, i[0], i[1], i[2]);
        const bool keep = inside(i, plo, phi);
        const float rho0 = g.rho[k];
#pragma unroll
        for (int a = 0; a < NDIM; a++) {
            if (i[a] < g.L[a] + N - 1 || i[a] > g.H[a] - N) continue;
            const long long st = gstride(g, a);
            float D = 0.0f;
#pragma unroll
            for (int l = 1; l <= N; l++) D += g.c[a][l - 1] * (p[k + l * st] - p[k - (l - 1) * st]);
            float *v = f.v[a] + s * g.ntot;
            v[k] = keep ? v[k] + g.dt * buoyancy(g, a, i[a], k, rho0) * D : 0.0f;
        }
    }
}

// ---------------------------------------------------------------------------
__global__ void k_inject_source(Grid g, Batch b, float *p, const float *stf, int it, float scale)
{
    const int s = blockIdx.x;
    const Stencil &st = b.src[s];
    const int n = st.cnt[0] * st.cnt[1] * st.cnt[2];
    const float amp = scale * stf[it];
    for (int t = threadIdx.x; t < n; t += blockDim.x) {
        const int a0 = t % st.cnt[0], r = t / st.cnt[0];
        const int a1 = r % st.cnt[1], a2 = r / st.cnt[1];
        const float w = st.w[0][a0] * st.w[1][a1] * st.w[2][a2];
        p[s * g.ntot + gidx(g, st.first[0] + a0, st.first[1] + a1, st.first[2] + a2)] += amp * w;
    }
}

__global__ void k_gather(Grid g, Batch b, const float *p, float *seis, const long long *seis_off,
                         int it)
{
    const int s = blockIdx.y;
    const int nr = b.rec_off[s + 1] - b.rec_off[s];
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= nr) return;
    const Stencil &st = b.rec[b.rec_off[s] + r];
    const float *ps = p + s * g.ntot;
    float sum = 0.0f;
    for (int a2 = 0; a2 < st.cnt[2]; a2++)
        for (int a1 = 0; a1 < st.cnt[1]; a1++)
            for (int a0 = 0; a0 < st.cnt[0]; a0++)
                sum += st.w[0][a0] * st.w[1][a1] * st.w[2][a2] *
                       ps[gidx(g, st.first[0] + a0, st.first[1] + a1, st.first[2] + a2)];
    seis[seis_off[s] + (long long)it * nr + r] = sum;
}

// Adjoint source (Algorithm 2): lp += kappa w_r res at the receiver stencils.
__global__ void k_adj_inject(Grid g, Batch b, float *lp, const float *res, const long long *seis_off,
                             int it)
{
    const int s = blockIdx.y;
    const int nr = b.rec_off[s + 1] - b.rec_off[s];
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= nr) return;
    const Stencil &st = b.rec[b.rec_off[s] + r];
    const float val = res[seis_off[s] + (long long)it * nr + r];
    float *ls = lp + s * g.ntot;
    for (int a2 = 0; a2 < st.cnt[2]; a2++)
        for (int a1 = 0; a1 < st.cnt[1]; a1++)
            for (int a0 = 0; a0 < st.cnt[0]; a0++) {
                const long long k = gidx(g, st.first[0] + a0, st.first[1] + a1, st.first[2] + a2);
                atomicAdd(ls + k, g.K[k] * st.w[0][a0] * st.w[1][a1] * st.w[2][a2] * val);
            }
}

// The same on the tile kernels' adjoint state (smi_slab.h).
__global__ void k_adj_inject_tile(Grid g, Batch b, Fields A, const float *res, const long long *seis_off, int it)
{
    const int s = blockIdx.y;
    const int nr = b.rec_off[s + 1] - b.rec_off[s];
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= nr) {
        if (r == 0) pdl_wait();
        return;
    }
    const Stencil &st = b.rec[b.rec_off[s] + r];
    const float val = res[seis_off[s] + (long long)it * nr + r];
    const int n0 = st.cnt[0], n1 = st.cnt[1], n2 = st.cnt[2];
    pdl_wait();
    pdl_trigger();
    for (int a2 = 0; a2 < n2; a2++)
        for (int a1 = 0; a1 < n1; a1++)
            for (int a0 = 0; a0 < n0; a0++) {
                const int z = st.first[0] + a0, x = st.first[1] + a1, y = st.first[2] + a2;
                const long long k = gidx(g, z, x, y);
                const float add = g.K[k] * st.w[0][a0] * st.w[1][a1] * st.w[2][a2] * val;
                atomicAdd(A.p + s * g.ntot + k, add);
                const int q = zslab_quad(g, z & ~3), jx = slab_row(g, 1, x);
                if (q >= 0)
                    atomicAdd(A.psiv[0] + s * g.slab_n[0] + q + (z & 3) + (long long)g.zp * (x + (long long)g.ne[1] * y),
                              g.cpa[0][z] * add);
                if (jx >= 0)
                    atomicAdd(A.psiv[1] + s * g.slab_n[1] + z + (long long)g.px * (jx + (long long)g.xrows * y),
                              g.cpa[1][x] * add);
                const int jy = g.ndim == 3 ? slab_row(g, 2, y) : -1;
                if (jy >= 0)
                    atomicAdd(A.psiv[2] + s * g.slab_n[2] + z + (long long)g.px * (x + (long long)g.ne[1] * jy),
                              g.cpa[2][y] * add);
            }
}

// Adjoint of the wavelet samples (the transpose of k_inject_source): the
// source of step it enters p^{it+1} as dt stf[it] w / dV, so its adjoint is
// dt / dV sum_w w pbar over the source stencil, with pbar = lambda_p / kappa
// (the library's adjoint pressure is kappa times the plain adjoint).  One
// block per shot; part[s][it] = the shot's sample, summed in FP64.
__global__ void k_src_adjoint(Grid g, Batch b, const float *lp, double *part, int nt, int it, double scale)
{
    __shared__ double red[kThreads];
    const int s = blockIdx.x;
    const Stencil &st = b.src[s];
    const int n = st.cnt[0] * st.cnt[1] * st.cnt[2];
    double acc = 0.0;
    for (int t = threadIdx.x; t < n; t += blockDim.x) {
        const int a0 = t % st.cnt[0], r = t / st.cnt[0];
        const int a1 = r % st.cnt[1], a2 = r / st.cnt[1];
        const long long k = gidx(g, st.first[0] + a0, st.first[1] + a1, st.first[2] + a2);
        const double w = (double)st.w[0][a0] * (double)st.w[1][a1] * (double)st.w[2][a2];
        acc += w * (double)lp[s * g.ntot + k] / (double)g.K[k];
    }
    red[threadIdx.x] = acc;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) part[(long long)s * nt + it] = scale * red[0];
}

// out[it] (+)= sum_s part[s][it], shots in order.
__global__ void k_sum_series(const double *part, int nshot, int nt, double *out, int accumulate)
{
    const int it = blockIdx.x * blockDim.x + threadIdx.x;
    if (it >= nt) return;
    double v = accumulate ? out[it] : 0.0;
    for (int s = 0; s < nshot; s++) v += part[(long long)s * nt + it];
    out[it] = v;
}

__global__ void k_to_float(const double *a, int n, float *out)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = (float)a[i];
}

// FP64 partial sums of a[i] * b[i], one per block (grid-stride; the
// partials are summed in block order afterwards, so the result does not
// depend on scheduling).
__global__ void k_dot(const float *a, const float *b, long long n, double *partials)
{
    __shared__ double red[kThreads];
    double acc = 0.0;
    for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < n;
         t += (long long)gridDim.x * blockDim.x)
        acc += (double)a[t] * (double)b[t];
    red[threadIdx.x] = acc;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) partials[blockIdx.x] = red[0];
}

// ---------------------------------------------------------------------------
// Boundary bands.  blockIdx.y = region r = 2 axis + side, blockIdx.z =
// shot; a thread moves kBandVals values of the region (stride 256, all
// loads issued before the stores).  One step of one shot holds fewer than
// 2^31 values (checked at set-up), so offsets are 32-bit.
constexpr int kBandVals = 4;

__global__ void k_band_absmax(Grid g, Fields f, Bands bd, unsigned *amax)
{
    const BandRegion R(bd, blockIdx.y);
    if (R.a >= g.ndim || R.n <= 0) return;
    const int s = blockIdx.z;
    const float *v = f.v[R.a] + (long long)s * g.ntot;
    float m = 0.0f;
#pragma unroll
    for (int q = 0; q < kBandVals; q++) {
        const int u = (blockIdx.x * kBandVals + q) * blockDim.x + threadIdx.x;
        if (u >= R.n) continue;
        int node, place;
        R.at(g, u, node, place);
        m = fmaxf(m, fabsf(v[node]));
    }
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0 && m > 0.0f) atomicMax(amax + s * 6 + blockIdx.y, __float_as_uint(m));
}

__global__ void k_band_save(Grid g, Fields f, Bands bd, int it, const unsigned *amax)
{
    pdl_wait();
    pdl_trigger();
    const BandRegion R(bd, blockIdx.y);
    if (R.a >= g.ndim || R.n <= 0) return;
    const int s = blockIdx.z;
    const float *v = f.v[R.a] + (long long)s * g.ntot;
    const long long b0 = (long long)s * bd.nt + it;
    float scale = 1.0f;
    if (bd.prec != SMI_PREC_F32) {
        scale = band_scale(bd, amax[s * 6 + blockIdx.y]);
        if (blockIdx.x == 0 && threadIdx.x == 0) bd.scale[b0 * 6 + blockIdx.y] = scale;
    }
    const float inv = band_inv(scale);
    float x[kBandVals];
    int place[kBandVals];
#pragma unroll
    for (int q = 0; q < kBandVals; q++) {
        const int u = (blockIdx.x * kBandVals + q) * blockDim.x + threadIdx.x;
        int node;
        R.at(g, min(u, R.n - 1), node, place[q]);
        x[q] = v[node];
    }
#pragma unroll
    for (int q = 0; q < kBandVals; q++) {
        const int u = (blockIdx.x * kBandVals + q) * blockDim.x + threadIdx.x;
        if (u < R.n) band_put(bd, b0 * bd.count + place[q], x[q], scale, inv);
    }
}

// Band of step it: sum_q w_q sample[first+q] over the samples that exist
// (before sample 0 the field is zero), or with one weight that sample alone.
// A thread takes kBandVals values and has the loads of all their samples in
// flight: a step reads 16 stored steps, which L2 holds from the step before.
template <int NT>
__global__ void k_band_restore(Grid g, Fields f, Bands bd, TimeWeights tw)
{
    pdl_wait();
    pdl_trigger();
    const BandRegion R(bd, blockIdx.y);
    if (R.a >= g.ndim || R.n <= 0) return;
    const int s = blockIdx.z;
    float *v = f.v[R.a] + (long long)s * g.ntot;
    int node[kBandVals], place[kBandVals];
#pragma unroll
    for (int q = 0; q < kBandVals; q++) {
        const int u = (blockIdx.x * kBandVals + q) * blockDim.x + threadIdx.x;
        R.at(g, min(u, R.n - 1), node[q], place[q]);
    }
    float x[kBandVals] = {};
#pragma unroll
    for (int t0 = 0; t0 < NT; t0 += 8) {
        constexpr int M = NT < 8 ? NT : 8;
        float y[M][kBandVals], wt[M];
#pragma unroll
        for (int t = 0; t < M; t++) {
            const int k = tw.first + t0 + t, kc = min(max(k, 0), tw.nsamp - 1);
            const long long b0 = (long long)s * bd.nt + kc;
            wt[t] = k == kc ? tw.w[t0 + t] : 0.0f;
            if (bd.prec != SMI_PREC_F32) wt[t] *= bd.scale[b0 * 6 + blockIdx.y];
#pragma unroll
            for (int q = 0; q < kBandVals; q++) y[t][q] = band_load(bd, b0 * bd.count + place[q], 1.0f);
        }
#pragma unroll
        for (int t = 0; t < M; t++)
#pragma unroll
            for (int q = 0; q < kBandVals; q++) x[q] = NT == 1 ? wt[t] * y[t][q] : x[q] + wt[t] * y[t][q];
    }
#pragma unroll
    for (int q = 0; q < kBandVals; q++) {
        const int u = (blockIdx.x * kBandVals + q) * blockDim.x + threadIdx.x;
        if (u < R.n) v[node[q]] = x[q];
    }
}

// ---------------------------------------------------------------------------
// Residual (mode 0: u - d, mode 1: d) and per-block partial sums of
// 1/2 (u - d)^2 in FP64 (Eq. objfwi).
__global__ void k_residual(const float *u, const float *d, long long n, int mode, float *res,
                           double *partials)
{
    __shared__ double red[kThreads];
    double acc = 0.0;
    for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < n;
         t += (long long)gridDim.x * blockDim.x) {
        const float r = u[t] - d[t];
        res[t] = mode == 0 ? r : d[t];
        acc += 0.5 * (double)r * (double)r;
    }
    red[threadIdx.x] = acc;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) partials[blockIdx.x] = red[0];
}

__global__ void k_sum_partials(const double *partials, int n, double *out)
{
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    double s = 0.0;
    for (int i = 0; i < n; i++) s += partials[i];
    *out += s;
}

// out[k] = the physical nodes of array k in the fields' padded layout.
__global__ void k_unpad(Grid g, const float *a, long long n, float *out)
{
    const int n0 = g.H[0] - g.L[0] + 1, n1 = g.H[1] - g.L[1] + 1;
    for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < n * g.nphys;
         t += (long long)gridDim.x * blockDim.x) {
        const long long k = t / g.nphys, u = t - k * g.nphys, q = u / n0;
        const int i0 = (int)(u - q * n0), i1 = (int)(q % n1), i2 = (int)(q / n1);
        out[t] = a[k * g.ntot + gidx(g, g.L[0] + i0, g.L[1] + i1, g.L[2] + i2)];
    }
}

// out[x] (+)= sum_s acc[s][x], shots added in order (deterministic).
__global__ void k_reduce_shots(const float *acc, long long n, int nshot, float *out, int accumulate)
{
    for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < n;
         t += (long long)gridDim.x * blockDim.x) {
        float s = accumulate ? out[t] : 0.0f;
        for (int k = 0; k < nshot; k++) s += acc[k * n + t];
        out[t] = s;
    }
}

// Normalised image (Sec. 2.3): per shot s the largest illumination ill_s,
// then out (+)= sum_s acc_s / (ill_s + 1e-3 max ill_s), shots in order.
// Illuminations are non-negative, so their bit patterns order as unsigned.
__global__ void k_shot_max(const float *ill, long long n, unsigned *mx)
{
    const int s = blockIdx.y;
    float m = 0.0f;
    for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < n;
         t += (long long)gridDim.x * blockDim.x)
        m = fmaxf(m, ill[s * n + t]);
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0 && m > 0.0f) atomicMax(mx + s, __float_as_uint(m));
}

__global__ void k_reduce_norm(const float *acc, const float *ill, long long n, int nshot, const unsigned *mx,
                              float *out, int accumulate)
{
    for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < n;
         t += (long long)gridDim.x * blockDim.x) {
        float s = accumulate ? out[t] : 0.0f;
        for (int k = 0; k < nshot; k++) s += acc[k * n + t] / (ill[k * n + t] + 1e-3f * __uint_as_float(mx[k]));
        out[t] = s;
    }
}

// dJ/dVp = 2 rho Vp dJ/dkappa with dJ/dkappa = -dt sum lp div v / kappa and
// kappa = rho Vp^2: -2 dt sum(lp div v) / Vp.
__global__ void k_finalize_grad(long long n, const float *vp, float dt, float *gr)
{
    for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < n;
         t += (long long)gridDim.x * blockDim.x)
        gr[t] = -2.0f * dt * gr[t] / vp[t];
}

// Density gradient (Eq. gradrhokappa, rho varied at fixed Vp).  Step it sets
// v^{it+1/2} = v^{it-1/2} - dt b (D p + psi) and nothing else of the step
// depends on b; with lambda_v = -b vbar and b = 2 / (rho_i + rho_{i+1}),
// each half node gives half of G = sum_it lambda_v (v^{it+1/2} - v^{it-1/2})
// to dJ/drho of both of its nodes (the b^2 of db/drho cancels the 1/b^2 of
// vbar dv/db).  k_rho_acc runs at the end of reverse step it, when vprev
// holds v^{it+1/2}, the source field v^{it-1/2} and the adjoint lambda_v of
// v^{it+1/2}: G_a += sum_s lambda_v (vprev - v), then vprev <- v.
// Four z-consecutive nodes per thread (float4): box.lo[0] is a multiple of
// 4 and the box's z width a multiple of 4 (the host widens the box; G is
// read only on the half nodes next to the physical domain, which the
// widened box always covers).
// Bound by the latency of its loads: one axis per blockIdx.y and the loads of
// two shots in flight at 4 blocks a SM (60 registers).  All axes in a thread
// ran in two and a half waves of fewer blocks; 6 and 8 blocks are slower (92.8,
// 93.3 ms), and so is a dependent launch (93.2).  90 x 110 x 100 + 10 layers, 2
// shots, 300 steps: a gradient 93.9 -> 91.2 ms.
__global__ void __launch_bounds__(kThreads, 4) k_rho_acc(Grid g, int nshot, Fields F, Fields A, RhoAcc r, IBox box)
{
    const int wq = (box.hi[0] - box.lo[0] + 1) >> 2;
    const int w1 = box.hi[1] - box.lo[1] + 1;
    const long long vol = (long long)wq * w1 * (box.hi[2] - box.lo[2] + 1);
    const int a = blockIdx.y;              // (selected, not indexed: an index would put the pointers on the stack)
    const float *const fv = a == 0 ? F.v[0] : (a == 1 ? F.v[1] : F.v[2]);
    const float *const av = a == 0 ? A.v[0] : (a == 1 ? A.v[1] : A.v[2]);
    float *const pr = a == 0 ? r.vprev[0] : (a == 1 ? r.vprev[1] : r.vprev[2]);
    float *const gr = a == 0 ? r.G[0] : (a == 1 ? r.G[1] : r.G[2]);
    for (long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x; q < vol;
         q += (long long)gridDim.x * blockDim.x) {
        int iq, i1, i2;
        if (vol < (1LL << 31)) {          // 32-bit division (uniform branch)
            const int qq = (int)q, rr = qq / wq;
            iq = qq - rr * wq;
            i1 = rr % w1;
            i2 = rr / w1;
        } else {
            const long long rr = q / wq;
            iq = (int)(q - rr * wq);
            i1 = (int)(rr % w1);
            i2 = (int)(rr / w1);
        }
        const long long k = gidx(g, box.lo[0] + 4 * iq, box.lo[1] + i1, box.lo[2] + i2);
        float4 *const G = reinterpret_cast<float4 *>(gr + k);
        float4 t = *G;
        float4 c = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        auto add = [&](const float4 &v, const float4 &l, const float4 &pv) {
            c.x += l.x * (pv.x - v.x);
            c.y += l.y * (pv.y - v.y);
            c.z += l.z * (pv.z - v.z);
            c.w += l.w * (pv.w - v.w);
        };
        auto ld = [](const float *x, long long i) { return *reinterpret_cast<const float4 *>(x + i); };
        int s = 0;
        for (; s + 2 <= nshot; s += 2) {
            const long long k0 = s * g.ntot + k, k1 = k0 + g.ntot;
            const float4 v0 = ld(fv, k0), l0 = ld(av, k0), p0 = ld(pr, k0);
            const float4 v1 = ld(fv, k1), l1 = ld(av, k1), p1 = ld(pr, k1);
            add(v0, l0, p0);
            add(v1, l1, p1);
            *reinterpret_cast<float4 *>(pr + k0) = v0;
            *reinterpret_cast<float4 *>(pr + k1) = v1;
        }
        if (s < nshot) {
            const long long k0 = s * g.ntot + k;
            const float4 v0 = ld(fv, k0);
            add(v0, ld(av, k0), ld(pr, k0));
            *reinterpret_cast<float4 *>(pr + k0) = v0;
        }
        t.x += c.x;
        t.y += c.y;
        t.z += c.z;
        t.w += c.w;
        *G = t;
    }
}

// Outputs of a gradient with a parametrisation family (Sec. 2.2).  acc =
// sum over shots and steps of lambda_p div v on the physical grid, so that
// dJ/dkappa = -dt acc / kappa; then
//   dJ/dVp|rho = 2 rho Vp dJ/dkappa,  dJ/drho|Vp = Vp^2 dJ/dkappa + buoyancy part,
// family 1 (Vp, rho): those two; family 2 (Vp, Ip = rho Vp):
//   dJ/dVp|Ip = dJ/dVp|rho - dJ/drho|Vp rho / Vp,  dJ/dIp|Vp = dJ/drho|Vp / Vp;
// logp: with respect to the logarithms (each times its parameter).
// g1 may alias acc.
__global__ void k_finalize_family(Grid g, const float *vp, const float *rho, const float *acc, RhoAcc r,
                                  int family, int logp, float *g1, float *g2)
{
    const int n0 = g.H[0] - g.L[0] + 1, n1 = g.H[1] - g.L[1] + 1;
    for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < g.nphys;
         t += (long long)gridDim.x * blockDim.x) {
        const int i0 = (int)(t % n0);
        const int i1 = (int)((t / n0) % n1);
        const int i2 = (int)(t / ((long long)n0 * n1));
        const long long k = gidx(g, i0 + g.L[0], i1 + g.L[1], i2 + g.L[2]);
        const float v = vp[t], d = rho[t], A0 = acc[t];
        float gb = 0.0f;
        for (int a = 0; a < g.ndim; a++) gb += r.G[a][k] + r.G[a][k - gstride(g, a)];
        float gv = -2.0f * g.dt * A0 / v;
        float gr = -g.dt * A0 / d + 0.5f * gb;
        if (family == 2) {
            gv -= gr * d / v;
            gr /= v;
        }
        if (logp) {
            gv *= v;
            gr *= family == 2 ? d * v : d;
        }
        g1[t] = gv;
        g2[t] = gr;
    }
}

// Free-surface mirrors and their transposes over the rows of nshot arrays
// (pitch px, stride floats a shot); thread (j, row, shot), j in 0..N fastest.
__global__ void k_free_surface(Grid g, float *f, long long rows, long long stride, int nshot, int op)
{
    const int N = g.N;
    const long long n = rows * nshot * (N + 1);
    const int L = g.L[0];
    for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < n;
         t += (long long)gridDim.x * blockDim.x) {
        const int j = (int)(t % (N + 1));
        const long long r = t / (N + 1);                 // shot * rows + row
        const long long s = r / rows, row = r - s * rows;
        float *c = f + s * stride + row * g.px;          // the z column of this (x, y)
        if (op == kFsMirrorV) {
            if (j < N) c[L - 1 - j] = c[L + j];
        } else if (op == kFsMirrorP) {
            if (j == 0) c[L] = 0.0f;
            else c[L - j] = -c[L + j];
        } else if (op == kFsFoldV) {
            if (j < N) {
                c[L + j] += c[L - 1 - j];
                c[L - 1 - j] = 0.0f;
            }
        } else {
            if (j == 0) {
                c[L] = 0.0f;
            } else {
                c[L + j] -= c[L - j];
                c[L - j] = 0.0f;
            }
        }
    }
}

__global__ void k_nonfinite(const float *x, long long n, unsigned *flag)
{
    bool bad = false;
    for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < n;
         t += (long long)gridDim.x * blockDim.x)
        bad |= !isfinite(x[t]);
    if (__syncthreads_or(bad) && threadIdx.x == 0) atomicOr(flag, 1u);
}

__global__ void k_extend_model(Grid g, const float *vp, const float *rho, int n1, int n2, int n3,
                               float *K, float *rho_e)
{
    for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < g.ntot;
         t += (long long)gridDim.x * blockDim.x) {
        const int i1 = (int)(t % g.px);
        const int i2 = (int)((t / g.px) % g.ne[1]);
        const int i3 = (int)(t / ((long long)g.px * g.ne[1]));
        // row padding: kappa 0, rho that of the last node (its own neighbour in the buoyancy)
        const bool pad = i1 >= g.ne[0];
        // free surface: the top layer mirrors the model about the surface node,
        // so that the transposed mirrors of the adjoint take no model ratio
        const int j1 = (g.freesurf && i1 < g.L[0]) ? min(g.L[0] - i1, n1 - 1) : min(max(i1 - g.L[0], 0), n1 - 1);
        const int j2 = min(max(i2 - g.L[1], 0), n2 - 1);
        const int j3 = min(max(i3 - g.L[2], 0), n3 - 1);
        const long long kp = (long long)j1 + (long long)n1 * ((long long)j2 + (long long)n2 * j3);
        const float r = rho[kp], c = vp[kp];
        rho_e[t] = r;
        K[t] = pad ? 0.0f : r * c * c;
    }
}

__global__ void k_minmax_init(unsigned *tmp)
{
    tmp[0] = 0x7f800000u;   // +inf
    tmp[1] = 0u;
}

// min/max of positive floats via their ordered bit patterns (NaN or <= 0
// entries force min to 0 so that the host rejects the model).
__global__ void k_minmax(const float *x, long long n, unsigned *tmp)
{
    unsigned lo = 0x7f800000u, hi = 0u;
    for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < n;
         t += (long long)gridDim.x * blockDim.x) {
        const float v = x[t];
        const unsigned u = (v > 0.0f && isfinite(v)) ? __float_as_uint(v) : 0u;
        lo = min(lo, u);
        hi = max(hi, u);
    }
    atomicMin(tmp, lo);
    atomicMax(tmp + 1, hi);
}

__global__ void k_minmax_out(const unsigned *tmp, float *out2)
{
    out2[0] = __uint_as_float(tmp[0]);
    out2[1] = __uint_as_float(tmp[1]);
}

__global__ void k_box_fill(Grid g, const int *ext, int nshot, int nt, int *tab)
{
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= (long long)nshot * (nt + 1)) return;
    const int s = (int)(t / (nt + 1)), n = (int)(t % (nt + 1)) - 1;
    int lo[3], hi[3];
    box_bounds(g, ext + 6 * s, n, lo, hi);
    for (int a = 0; a < 3; a++) {
        tab[t * 6 + a] = lo[a];
        tab[t * 6 + 3 + a] = hi[a];
    }
}

__global__ void k_box_table(Grid g, const int *ext, int n0, int count, int *lo, int *hi)
{
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= count) return;
    box_bounds(g, ext, n0 + c, lo + 3 * c, hi + 3 * c);
}

inline cudaStream_t S(const LaunchCtx &lc) { return static_cast<cudaStream_t>(lc.stream); }

inline int blocks_for(long long n)
{
    long long b = (n + kThreads - 1) / kThreads;
    if (b < 1) b = 1;
    return (int)(b < kMaxBlocksX ? b : kMaxBlocksX);
}

}  // namespace

// ---------------------------------------------------------------------------
#define SMI_DISPATCH(KERNEL, GRID, ...)                                                    \
    do {                                                                                   \
        if (g.ndim == 2 && g.N == 2) KERNEL<2, 2><<<GRID, kThreads, 0, S(lc)>>>(__VA_ARGS__); \
        else if (g.ndim == 2 && g.N == 4) KERNEL<2, 4><<<GRID, kThreads, 0, S(lc)>>>(__VA_ARGS__); \
        else if (g.ndim == 3 && g.N == 2) KERNEL<3, 2><<<GRID, kThreads, 0, S(lc)>>>(__VA_ARGS__); \
        else KERNEL<3, 4><<<GRID, kThreads, 0, S(lc)>>>(__VA_ARGS__);                       \
        ++*lc.launches;                                                                    \
    } while (0)

void launch_fwd_v(const LaunchCtx &lc, const Grid &g, const Batch &b, Fields f, int it, long long work)
{
    dim3 grid(blocks_for(work), b.nshot);
    SMI_DISPATCH(k_fwd_v, grid, g, b, f, it);
}

void launch_fwd_p(const LaunchCtx &lc, const Grid &g, const Batch &b, Fields f, int it, long long work)
{
    dim3 grid(blocks_for(work), b.nshot);
    SMI_DISPATCH(k_fwd_p, grid, g, b, f, it);
}

void launch_adj_v(const LaunchCtx &lc, const Grid &g, const Batch &b, Fields f, int m, long long work)
{
    dim3 grid(blocks_for(work), b.nshot);
    SMI_DISPATCH(k_adj_v, grid, g, b, f, m);
}

void launch_adj_p(const LaunchCtx &lc, const Grid &g, const Batch &b, Fields f, int m, long long work)
{
    dim3 grid(blocks_for(work), b.nshot);
    SMI_DISPATCH(k_adj_p, grid, g, b, f, m);
}

void launch_recon_p(const LaunchCtx &lc, const Grid &g, const Batch &b, Fields f, const float *lp,
                    float *acc, int mode, const float *stf, int it, float src_scale, long long work)
{
    dim3 grid(blocks_for(work), b.nshot);
    SMI_DISPATCH(k_recon_p, grid, g, b, f, lp, acc, mode, stf, it, src_scale);
}

void launch_recon_v(const LaunchCtx &lc, const Grid &g, const Batch &b, Fields f, int it, long long work)
{
    dim3 grid(blocks_for(work), b.nshot);
    SMI_DISPATCH(k_recon_v, grid, g, b, f, it);
}

void launch_inject_source(const LaunchCtx &lc, const Grid &g, const Batch &b, float *p,
                          const float *stf, int it, float scale)
{
    k_inject_source<<<b.nshot, 128, 0, S(lc)>>>(g, b, p, stf, it, scale);
    ++*lc.launches;
}

void launch_gather(const LaunchCtx &lc, const Grid &g, const Batch &b, const float *p, float *seis,
                   const long long *seis_off, int nt, int it)
{
    (void)nt;
    dim3 grid((b.max_rec + 127) / 128, b.nshot);
    k_gather<<<grid, 128, 0, S(lc)>>>(g, b, p, seis, seis_off, it);
    ++*lc.launches;
}

void launch_adj_inject(const LaunchCtx &lc, const Grid &g, const Batch &b, float *lp, const float *res,
                       const long long *seis_off, int nt, int it)
{
    (void)nt;
    dim3 grid((b.max_rec + 127) / 128, b.nshot);
    k_adj_inject<<<grid, 128, 0, S(lc)>>>(g, b, lp, res, seis_off, it);
    ++*lc.launches;
}

void launch_adj_inject_tile(const LaunchCtx &lc, const Grid &g, const Batch &b, Fields A, const float *res,
                            const long long *seis_off, int it)
{
    launch_pdl(lc, k_adj_inject_tile, dim3((b.max_rec + 127) / 128, b.nshot), 128, 0, g, b, A, res, seis_off, it);
}

// Band kernels: x = chunks of the largest region, y = region, z = shot.
static dim3 band_grid(const Bands &bd, int nshot)
{
    long long nmax = 0;
    for (int a = 0; a < 3; a++)
        for (int sd = 0; sd < 2; sd++) {
            long long n = 1;
            for (int b = 0; b < 3; b++) n *= std::max(0, bd.hi[a][sd][b] - bd.lo[a][sd][b] + 1);
            nmax = std::max(nmax, n);
        }
    return dim3((unsigned)std::max<long long>(1, (nmax + kThreads * kBandVals - 1) / (kThreads * kBandVals)), 6, nshot);
}

void launch_save_bands(const LaunchCtx &lc, const Grid &g, const Batch &b, Fields f, Bands bd, int it,
                       unsigned *absmax_tmp, bool have_max)
{
    const dim3 grid = band_grid(bd, b.nshot);
    if (bd.prec != SMI_PREC_F32 && !have_max) {
        cudaMemsetAsync(absmax_tmp, 0, sizeof(unsigned) * 6 * b.nshot, S(lc));
        k_band_absmax<<<grid, kThreads, 0, S(lc)>>>(g, f, bd, absmax_tmp);
        ++*lc.launches;
    }
    launch_pdl(lc, k_band_save, grid, kThreads, 0, g, f, bd, it, absmax_tmp);
}

void launch_restore_bands_interp(const LaunchCtx &lc, const Grid &g, const Batch &b, Fields f, Bands bd,
                                 const TimeWeights &tw)
{
    bool one = true;                           // a step on a stored sample
    for (int q = 1; q < 2 * kTimeR; q++) one = one && tw.w[q] == 0.0f;
    if (one) launch_pdl(lc, k_band_restore<1>, band_grid(bd, b.nshot), kThreads, 0, g, f, bd, tw);
    else launch_pdl(lc, k_band_restore<2 * kTimeR>, band_grid(bd, b.nshot), kThreads, 0, g, f, bd, tw);
}

void launch_restore_bands(const LaunchCtx &lc, const Grid &g, const Batch &b, Fields f, Bands bd, int it)
{
    TimeWeights tw{};
    tw.first = it;
    tw.nsamp = bd.nt;
    tw.w[0] = 1.0f;
    launch_restore_bands_interp(lc, g, b, f, bd, tw);
}

void launch_residual(const LaunchCtx &lc, const float *seis, const float *dobs, long long n, int mode,
                     float *res, double *partials, int npart)
{
    k_residual<<<npart, kThreads, 0, S(lc)>>>(seis, dobs, n, mode, res, partials);
    ++*lc.launches;
}

void launch_src_adjoint(const LaunchCtx &lc, const Grid &g, const Batch &b, const float *lp, double *part, int nt,
                        int it, double scale)
{
    k_src_adjoint<<<b.nshot, kThreads, 0, S(lc)>>>(g, b, lp, part, nt, it, scale);
    ++*lc.launches;
}

void launch_sum_series(const LaunchCtx &lc, const double *part, int nshot, int nt, double *out, int accumulate)
{
    k_sum_series<<<(nt + kThreads - 1) / kThreads, kThreads, 0, S(lc)>>>(part, nshot, nt, out, accumulate);
    ++*lc.launches;
}

void launch_to_float(const LaunchCtx &lc, const double *a, int n, float *out)
{
    k_to_float<<<(n + kThreads - 1) / kThreads, kThreads, 0, S(lc)>>>(a, n, out);
    ++*lc.launches;
}

void launch_dot(const LaunchCtx &lc, const float *a, const float *b, long long n, double *partials, int npart)
{
    k_dot<<<npart, kThreads, 0, S(lc)>>>(a, b, n, partials);
    ++*lc.launches;
}

void launch_sum_partials(const LaunchCtx &lc, const double *partials, int npart, double *out)
{
    k_sum_partials<<<1, 32, 0, S(lc)>>>(partials, npart, out);
    ++*lc.launches;
}

void launch_unpad(const LaunchCtx &lc, const Grid &g, const float *a, size_t n, float *out)
{
    k_unpad<<<blocks_for(g.nphys * (long long)n), kThreads, 0, S(lc)>>>(g, a, (long long)n, out);
    ++*lc.launches;
}

void launch_reduce_shots(const LaunchCtx &lc, const Grid &g, const float *acc, int nshot, float *out,
                         int accumulate)
{
    k_reduce_shots<<<blocks_for(g.nphys), kThreads, 0, S(lc)>>>(acc, g.nphys, nshot, out, accumulate);
    ++*lc.launches;
}

void launch_reduce_norm(const LaunchCtx &lc, const Grid &g, const float *acc, int nshot, unsigned *mx, float *out,
                        int accumulate)
{
    const float *ill = acc + (long long)nshot * g.nphys;
    cudaMemsetAsync(mx, 0, sizeof(unsigned) * nshot, S(lc));
    k_shot_max<<<dim3(blocks_for(g.nphys), nshot), kThreads, 0, S(lc)>>>(ill, g.nphys, mx);
    k_reduce_norm<<<blocks_for(g.nphys), kThreads, 0, S(lc)>>>(acc, ill, g.nphys, nshot, mx, out, accumulate);
    *lc.launches += 2;
}

void launch_finalize_grad(const LaunchCtx &lc, long long n, const float *vp, float dt, float *gr)
{
    k_finalize_grad<<<blocks_for(n), kThreads, 0, S(lc)>>>(n, vp, dt, gr);
    ++*lc.launches;
}

void launch_rho_acc(const LaunchCtx &lc, const Grid &g, int nshot, Fields F, Fields A, RhoAcc r, IBox box)
{
    long long vol = 1;
    for (int a = 0; a < 3; a++) vol *= std::max(0, box.hi[a] - box.lo[a] + 1);
    if (vol == 0) return;
    box.lo[0] &= ~3;                       // whole float4 quads; px is a multiple of 8
    box.hi[0] |= 3;
    const long long quads = (long long)((box.hi[0] - box.lo[0] + 1) >> 2) * (box.hi[1] - box.lo[1] + 1) *
                            (box.hi[2] - box.lo[2] + 1);
    k_rho_acc<<<dim3(blocks_for(quads), g.ndim), kThreads, 0, S(lc)>>>(g, nshot, F, A, r, box);
    ++*lc.launches;
}

void launch_finalize_family(const LaunchCtx &lc, const Grid &g, const float *vp, const float *rho, const float *acc,
                            RhoAcc r, int family, int logp, float *g1, float *g2)
{
    k_finalize_family<<<blocks_for(g.nphys), kThreads, 0, S(lc)>>>(g, vp, rho, acc, r, family, logp, g1, g2);
    ++*lc.launches;
}

static void free_surface_rows(const LaunchCtx &lc, const Grid &g, float *f, long long rows, long long stride,
                              int nshot, int op)
{
    const long long n = rows * nshot * (g.N + 1);
    k_free_surface<<<blocks_for(n), kThreads, 0, S(lc)>>>(g, f, rows, stride, nshot, op);
    ++*lc.launches;
}

void launch_free_surface(const LaunchCtx &lc, const Grid &g, float *f, int nshot, int op)
{
    if (g.freesurf) free_surface_rows(lc, g, f, (long long)g.ne[1] * g.ne[2], g.ntot, nshot, op);
}

void launch_free_surface_fold_tile(const LaunchCtx &lc, const Grid &g, Fields A, int nshot)
{
    if (!g.freesurf) return;
    launch_free_surface(lc, g, A.p, nshot, kFsFoldP);
    free_surface_rows(lc, g, A.psiv[1], (long long)g.xrows * g.ne[2], g.slab_n[1], nshot, kFsFoldP);
    if (g.ndim == 3) free_surface_rows(lc, g, A.psiv[2], (long long)g.ne[1] * g.S, g.slab_n[2], nshot, kFsFoldP);
}

void launch_nonfinite(const LaunchCtx &lc, const float *x, long long n, unsigned *flag)
{
    k_nonfinite<<<blocks_for(n), kThreads, 0, S(lc)>>>(x, n, flag);
    ++*lc.launches;
}

void launch_extend_model(const LaunchCtx &lc, const Grid &g, const float *vp, const float *rho, int n1,
                         int n2, int n3, float *K, float *rho_e)
{
    k_extend_model<<<blocks_for(g.ntot), kThreads, 0, S(lc)>>>(g, vp, rho, n1, n2, n3, K, rho_e);
    ++*lc.launches;
}

void launch_minmax(const LaunchCtx &lc, const float *vp, long long n, float *out2, unsigned *tmp)
{
    k_minmax_init<<<1, 1, 0, S(lc)>>>(tmp);
    k_minmax<<<blocks_for(n), kThreads, 0, S(lc)>>>(vp, n, tmp);
    k_minmax_out<<<1, 1, 0, S(lc)>>>(tmp, out2);
    *lc.launches += 3;
}

void launch_zero(const LaunchCtx &lc, void *ptr, size_t bytes)
{
    cudaMemsetAsync(ptr, 0, bytes, S(lc));
}

void launch_box_fill(const LaunchCtx &lc, const Grid &g, const int *ext, int nshot, int nt, int *tab)
{
    const long long n = (long long)nshot * (nt + 1);
    k_box_fill<<<(unsigned)((n + 127) / 128), 128, 0, S(lc)>>>(g, ext, nshot, nt, tab);
    ++*lc.launches;
}

void launch_box_table(const LaunchCtx &lc, const Grid &g, const int *ext, int n0, int count, int *lo,
                      int *hi)
{
    k_box_table<<<(count + 127) / 128, 128, 0, S(lc)>>>(g, ext, n0, count, lo, hi);
    ++*lc.launches;
}

}  // namespace smi
