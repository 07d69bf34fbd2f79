// smi_band.h -- boundary bands (Sec. 4.2): the regions of one step's stored
// velocities, and the parts of saving and restoring them that the 3D tile
// kernels run after their own work.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "smi_internal.h"
#include "smi_stencil3d.h"

#ifdef __CUDACC__
namespace smi {

struct BandRegion {
    int a, sd, w0, w1, n, off, s0, s1;
    const int *lo;
    unsigned m0, m1;                  // u / w0 and q / w1 by multiply-high (band_divisor)
    int l0, l1;
    __device__ __forceinline__ BandRegion(const Bands &bd, int r)
    {
        a = r >> 1;
        sd = r & 1;
        lo = bd.lo[a][sd];
        const int *hi = bd.hi[a][sd];
        w0 = hi[0] - lo[0] + 1;
        w1 = hi[1] - lo[1] + 1;
        n = w0 > 0 && w1 > 0 ? w0 * w1 * max(0, hi[2] - lo[2] + 1) : 0;
        s0 = bd.sw[a][sd][0];
        s1 = bd.sw[a][sd][1];
        off = (int)bd.off[a][sd];
        m0 = bd.dm[a][sd][0];
        l0 = bd.dl[a][sd][0];
        m1 = bd.dm[a][sd][1];
        l1 = bd.dl[a][sd][1];
    }
    // flat field index of value u of the region, and its place in a stored step
    __device__ __forceinline__ void at(const Grid &g, int u, int &node, int &place) const
    {
        const unsigned uu = (unsigned)u;
        const unsigned q = (__umulhi(m0, uu) + uu) >> l0;
        const unsigned q1 = (__umulhi(m1, q) + q) >> l1;
        const int z = u - (int)q * w0, x = (int)q - (int)q1 * w1, y = (int)q1;
        node = (lo[0] + z) + g.px * ((lo[1] + x) + g.ne[1] * (lo[2] + y));
        place = off + z + s0 * (x + s1 * y);
    }
};

// Every CTA takes its share of the values of one region after another.
template <class F> __device__ __forceinline__ void for_band_values(const Grid &g, const Bands &bd, int nshot, F f)
{
    for (int s = 0; s < nshot; s++)
        for (int r = 0; r < 2 * g.ndim; r++) {
            const BandRegion R(bd, r);
            for (int u = blockIdx.x * blockDim.x + threadIdx.x; u < R.n; u += gridDim.x * blockDim.x) f(s, r, R, u);
        }
}

// Stores x at place o; 16-bit storage scaled per (step, axis, side): the
// largest magnitude maps to 2^14 (FP16) or 1 (BF16).  inv = 1 / scale (0 when
// that would overflow: early steps, which divide).
__device__ __forceinline__ void band_put(const Bands &bd, long long o, float x, float scale, float inv)
{
    if (bd.prec == SMI_PREC_F32) {
        static_cast<float *>(bd.data)[o] = x;
        return;
    }
    float y = x * inv;
    if (inv == 0.0f) y = scale > 0.0f ? x / scale : 0.0f;
    if (bd.prec == SMI_PREC_F16) static_cast<__half *>(bd.data)[o] = __float2half_rn(y);
    else static_cast<__nv_bfloat16 *>(bd.data)[o] = __float2bfloat16_rn(y);
}
__device__ __forceinline__ float band_scale(const Bands &bd, unsigned mx)
{
    return __uint_as_float(mx) / (bd.prec == SMI_PREC_F16 ? 16384.0f : 1.0f);
}
__device__ __forceinline__ float band_inv(float scale) { return scale < 1e-36f ? 0.0f : __frcp_rn(scale); }

// The band of the velocities in f as stored sample sv.sample, or (find) their
// largest magnitude per (shot, axis, side) into sv.amax.
__device__ __forceinline__ void save_tail(const Grid &g, int nshot, const Fields &f, const Save3 &sv)
{
    const Bands &bd = sv.bd;
    const int first = blockIdx.x * blockDim.x + threadIdx.x, stride = gridDim.x * blockDim.x;
    for (int s = 0; s < nshot; s++)
        for (int r = 0; r < 2 * g.ndim; r++) {
            const BandRegion R(bd, r);
            const float *v = f.v[R.a] + (long long)s * g.ntot;
            int node, place;
            if (sv.find) {
                float m = 0.0f;
                for (int u = first; u < R.n; u += stride) {
                    R.at(g, u, node, place);
                    m = fmaxf(m, fabsf(v[node]));
                }
                const unsigned mx = __reduce_max_sync(0xffffffffu, __float_as_uint(m));
                if ((threadIdx.x & 31) == 0 && mx) atomicMax(sv.amax + s * 6 + r, mx);
                continue;
            }
            const long long b0 = (long long)s * bd.nt + sv.sample;
            float scale = 1.0f;
            if (bd.prec != SMI_PREC_F32) {
                scale = band_scale(bd, sv.amax[s * 6 + r]);
                if (first == 0) bd.scale[b0 * 6 + r] = scale;
            }
            const float inv = band_inv(scale);
            for (int u = first; u < R.n; u += stride) {
                R.at(g, u, node, place);
                band_put(bd, b0 * bd.count + place, v[node], scale, inv);
            }
        }
}

// Stored value o, rescaled.
__device__ __forceinline__ float band_load(const Bands &bd, long long o, float scale)
{
    if (bd.prec == SMI_PREC_F32) return static_cast<const float *>(bd.data)[o];
    if (bd.prec == SMI_PREC_F16) return __half2float(static_cast<const __half *>(bd.data)[o]) * scale;
    return __bfloat162float(static_cast<const __nv_bfloat16 *>(bd.data)[o]) * scale;
}

// The stored band of step rs.it into the source velocities rs.v.
__device__ __forceinline__ void restore_tail(const Grid &g, int nshot, const Restore3 &rs)
{
    const Bands &bd = rs.bd;
    for_band_values(g, bd, nshot, [&](int s, int r, const BandRegion &R, int u) {
        const long long b0 = (long long)s * bd.nt + rs.it;
        const float sc = bd.prec == SMI_PREC_F32 ? 1.0f : bd.scale[b0 * 6 + r];
        int node, place;
        R.at(g, u, node, place);
        rs.v[R.a][(long long)s * g.ntot + node] = band_load(bd, b0 * bd.count + place, sc);
    });
}

// Receivers' samples of the pressure p.
__device__ __forceinline__ void gather_tail(const Grid &g, const Batch &b, const float *p, const Gather3 &ga)
{
    for (int s = 0; s < b.nshot; s++) {
        const int nr = b.rec_off[s + 1] - b.rec_off[s];
        for (int r = blockIdx.x * blockDim.x + threadIdx.x; r < nr; r += gridDim.x * blockDim.x) {
            const Stencil &st = b.rec[b.rec_off[s] + r];
            const float *ps = p + (long long)s * g.ntot;
            float sum = 0.0f;
            for (int a2 = 0; a2 < st.cnt[2]; a2++)
                for (int a1 = 0; a1 < st.cnt[1]; a1++)
                    for (int a0 = 0; a0 < st.cnt[0]; a0++)
                        sum += st.w[0][a0] * st.w[1][a1] * st.w[2][a2] *
                               ps[st.first[0] + a0 +
                                  (long long)g.px * (st.first[1] + a1 + (long long)g.ne[1] * (st.first[2] + a2))];
            ga.seis[ga.off[s] + (long long)ga.it * nr + r] = sum;
        }
    }
}

}  // namespace smi
#endif
