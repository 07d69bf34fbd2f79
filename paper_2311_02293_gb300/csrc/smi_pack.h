// smi_pack.h -- quads of four z nodes in packed FP32 arithmetic (f32x2), for
// the tile kernels.
#pragma once

#include <cuda_runtime.h>

#include "smi_internal.h"
#include "smi_slab.h"

namespace smi {

// Quads of FP32 as two packed pairs (each lane rounds like a scalar
// operation): half the instructions, and a 128-bit load is a quad as it is.
typedef unsigned long long P2;
__device__ __forceinline__ P2 pack(float a, float b)
{
    P2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void unpack(P2 p, float &a, float &b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(p)); }
__device__ __forceinline__ P2 add2(P2 a, P2 b)
{
    P2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ P2 sub2(P2 a, P2 b)
{
    P2 r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ P2 mul2(P2 a, P2 b)
{
    P2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ P2 fma2(P2 a, P2 b, P2 c)
{
    P2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
struct Q4 {
    P2 a, b;
};
__device__ __forceinline__ Q4 ldq(const float *p)
{
    const ulonglong2 t = *reinterpret_cast<const ulonglong2 *>(p);
    return {t.x, t.y};
}
__device__ __forceinline__ void stq(float *p, const Q4 &q) { *reinterpret_cast<ulonglong2 *>(p) = make_ulonglong2(q.a, q.b); }
__device__ __forceinline__ Q4 quad(const float (&v)[4]) { return {pack(v[0], v[1]), pack(v[2], v[3])}; }
__device__ __forceinline__ Q4 zeroq() { return {0ull, 0ull}; }
__device__ __forceinline__ void split(const Q4 &q, float (&v)[4])
{
    unpack(q.a, v[0], v[1]);
    unpack(q.b, v[2], v[3]);
}
__device__ __forceinline__ Q4 addq(const Q4 &x, const Q4 &y) { return {add2(x.a, y.a), add2(x.b, y.b)}; }
__device__ __forceinline__ Q4 subq(const Q4 &x, const Q4 &y) { return {sub2(x.a, y.a), sub2(x.b, y.b)}; }
__device__ __forceinline__ Q4 mulq(const Q4 &x, const Q4 &y) { return {mul2(x.a, y.a), mul2(x.b, y.b)}; }
__device__ __forceinline__ Q4 fmaq(const Q4 &x, const Q4 &y, const Q4 &z) { return {fma2(x.a, y.a, z.a), fma2(x.b, y.b, z.b)}; }
// D + c (x - y)
__device__ __forceinline__ Q4 tap(const Q4 &D, float c, const Q4 &x, const Q4 &y)
{
    const P2 cc = pack(c, c);
    return {fma2(cc, sub2(x.a, y.a), D.a), fma2(cc, sub2(x.b, y.b), D.b)};
}
// num / (r0 + r1) as reciprocal and product.  The reciprocal is PTX's
// rcp.approx.ftz.f32, which the PTX ISA documents to within 1 ulp; with the
// product about 1.5 ulp, far below the FP32 scheme error.  Its operand is a sum
// of two densities, positive normal numbers.
__device__ __forceinline__ float rcpf(float x)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ Q4 buoyq(const Q4 &num, const Q4 &r0, const Q4 &r1)
{
    float d[4];
    split(addq(r0, r1), d);
#pragma unroll
    for (int r = 0; r < 4; r++) d[r] = rcpf(d[r]);
    return mulq(num, quad(d));
}
// Brings a line that a later plane reads towards the L2 cache.
__device__ __forceinline__ void prefetch_l2(const float *p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }
__device__ __forceinline__ void window(float (&W)[12], const float *row)
{
#pragma unroll
    for (int k = 0; k < 3; k++) {
        float v[4];
        split(ldq(row + 4 * k), v);
#pragma unroll
        for (int r = 0; r < 4; r++) W[4 * k + r] = v[r];
    }
}
// D along z of the middle quad of a window, p nodes to v nodes (UP) or back.
template <int N, bool UP> __device__ __forceinline__ Q4 dz4(const Grid &g, const float (&W)[12])
{
    float D[4];
#pragma unroll
    for (int r = 0; r < 4; r++) {
        float d = 0.f;
#pragma unroll
        for (int l = 1; l <= N; l++)
            d += g.c[0][l - 1] * (UP ? W[4 + r + l] - W[4 + r - l + 1] : W[4 + r + l - 1] - W[4 + r - l]);
        D[r] = d;
    }
    return quad(D);
}

// m <- B m + A x over the quad.
__device__ __forceinline__ void recur4(const float (&B)[4], const float (&A)[4], float (&m)[4], const Q4 &x)
{
    float v[4];
    split(x, v);
#pragma unroll
    for (int r = 0; r < 4; r++) m[r] = slab_recur(B[r], m[r], A[r], v[r]);
}
__device__ __forceinline__ void recur1(float B, float A, float (&m)[4], const Q4 &x)
{
    const float Bq[4] = {B, B, B, B}, Aq[4] = {A, A, A, A};
    recur4(Bq, Aq, m, x);
}
// v - b m
__device__ __forceinline__ Q4 sub_prod(const Q4 &v, const Q4 &b, const float (&m)[4])
{
    float x[4], c[4];
    split(v, x);
    split(b, c);
#pragma unroll
    for (int r = 0; r < 4; r++) x[r] = __fmaf_rn(-c[r], m[r], x[r]);
    return quad(x);
}
// Zero where z.
__device__ __forceinline__ Q4 clear_if(const Q4 &q, const bool (&z)[4])
{
    float x[4];
    split(q, x);
#pragma unroll
    for (int r = 0; r < 4; r++) x[r] = z[r] ? 0.f : x[r];
    return quad(x);
}

// Largest magnitude of the quad's nodes in mask, over the warp.
__device__ __forceinline__ unsigned warp_max(const Q4 &q, unsigned mask)
{
    float v[4], m = 0.0f;
    split(q, v);
#pragma unroll
    for (int r = 0; r < 4; r++) m = mask >> r & 1u ? fmaxf(m, fabsf(v[r])) : m;
    return __reduce_max_sync(0xffffffffu, __float_as_uint(m));
}

}  // namespace smi
