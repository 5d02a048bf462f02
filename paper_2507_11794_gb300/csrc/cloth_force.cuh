// What the kernels that evaluate spring forces share: packed FP32x2
// arithmetic, the force law on pairs of nodes, and programmatic launches.
#pragma once

#include <utility>

#include "cloth_internal.h"

namespace {

constexpr unsigned FULL = 0xffffffffu;

// Programmatic dependent launch: each kernel of a substep lets the next one
// be launched once all its CTAs are running (launch_dependents), and waits
// for the previous one to complete, with its writes visible, before it
// touches any state (wait).  The next kernel's launch and CTA start-up then
// overlap this kernel's tail instead of following it.
#ifndef CLOTH_PDL
#define CLOTH_PDL 1
#endif
__device__ __forceinline__ void pdl_wait()
{
#if CLOTH_PDL
    asm volatile("griddepcontrol.wait;" ::: "memory");
#endif
}
__device__ __forceinline__ void pdl_launch_dependents()
{
#if CLOTH_PDL
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
#endif
}
// Packed FP32x2 arithmetic as explicitly rounded PTX instructions (add.rn,
// mul.rn, fma.rn on .f32x2).  Each is one IEEE operation per component that
// no optimizer fuses or reorders, so a node's arithmetic is the same whichever
// copy of the unrolled row loop computes it; with the CUDA 13.0 packed
// intrinsics (__fadd2_rn, __fmul2_rn, __ffma2_rn) the four copies of the loop
// gave results one ulp apart, so a cloth's bits depended on its strip height.
__device__ __forceinline__ float2 add2(float2 a, float2 b)
{
    float2 r;
    asm("{.reg .b64 x, y, d;\n\tmov.b64 x, {%2, %3};\n\tmov.b64 y, {%4, %5};\n\tadd.rn.f32x2 d, x, y;\n\t"
        "mov.b64 {%0, %1}, d;}"
        : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return r;
}
__device__ __forceinline__ float2 mul2(float2 a, float2 b)
{
    float2 r;
    asm("{.reg .b64 x, y, d;\n\tmov.b64 x, {%2, %3};\n\tmov.b64 y, {%4, %5};\n\tmul.rn.f32x2 d, x, y;\n\t"
        "mov.b64 {%0, %1}, d;}"
        : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return r;
}
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c)
{
    float2 r;
    asm("{.reg .b64 x, y, z, d;\n\tmov.b64 x, {%2, %3};\n\tmov.b64 y, {%4, %5};\n\tmov.b64 z, {%6, %7};\n\t"
        "fma.rn.f32x2 d, x, y, z;\n\tmov.b64 {%0, %1}, d;}"
        : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
    return r;
}
// a - b, exact as one rounding: fma(b, -1, a)
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return fma2(b, make_float2(-1.0f, -1.0f), a); }
__device__ __forceinline__ float2 bc(float s) { return make_float2(s, s); }

struct Node2 {  // two nodes (A = .x, B = .y)
    float2 px, py, pz, vx, vy, vz;
};
struct Vec2 {  // one 3-vector per node of the pair
    float2 x, y, z;
};

__device__ __forceinline__ Vec2 vadd(Vec2 a, Vec2 b) { return {add2(a.x, b.x), add2(a.y, b.y), add2(a.z, b.z)}; }
__device__ __forceinline__ Vec2 vsub(Vec2 a, Vec2 b) { return {sub2(a.x, b.x), sub2(a.y, b.y), sub2(a.z, b.z)}; }

__device__ __forceinline__ float2 shfl_down2(float2 v, int d)
{
    return make_float2(__shfl_down_sync(FULL, v.x, d), __shfl_down_sync(FULL, v.y, d));
}
__device__ __forceinline__ float2 shfl_up2(float2 v, int d)
{
    return make_float2(__shfl_up_sync(FULL, v.x, d), __shfl_up_sync(FULL, v.y, d));
}
// Hooke's law plus damping along the spring (Algorithm 1) for the pair:
// d = q - p, F_p = (ks (|d| - L0) + kd (v_q - v_p).d / |d|) d / |d|, written
// as F_p = s d with s = (ks (|d| - L0) + kd il (v_q - v_p).d) il, il = 1/|d|
// (zero force for |d|^2 <= 1e-24).
// From the differences d = q - p (dx, dy, dz) and v_q - v_p (ux, uy, uz):
// spring_scale gives s, spring2d the force.
__device__ __forceinline__ float2 spring_scale(float2 dx, float2 dy, float2 dz, float2 ux, float2 uy, float2 uz,
                                               float2 ks, float2 kd, float L0)
{
    const float2 l2 = fma2(dz, dz, fma2(dy, dy, mul2(dx, dx)));
    float2 il;
    il.x = l2.x > 1e-24f ? rsqrtf(l2.x) : 0.0f;
    il.y = l2.y > 1e-24f ? rsqrtf(l2.y) : 0.0f;
    const float2 dvd = fma2(uz, dz, fma2(uy, dy, mul2(ux, dx)));
    const float2 e = fma2(l2, il, bc(-L0));  // |d| - L0
    return mul2(fma2(mul2(kd, il), dvd, mul2(ks, e)), il);
}
__device__ __forceinline__ Vec2 spring2d(float2 dx, float2 dy, float2 dz, float2 ux, float2 uy, float2 uz, float2 ks,
                                         float2 kd, float L0)
{
    const float2 sc = spring_scale(dx, dy, dz, ux, uy, uz, ks, kd, L0);
    return {mul2(sc, dx), mul2(sc, dy), mul2(sc, dz)};
}
__device__ __forceinline__ Vec2 spring2(const Node2 &P, const Node2 &Q, float2 ks, float2 kd, float L0)
{
    return spring2d(sub2(Q.px, P.px), sub2(Q.py, P.py), sub2(Q.pz, P.pz), sub2(Q.vx, P.vx), sub2(Q.vy, P.vy),
                    sub2(Q.vz, P.vz), ks, kd, L0);
}
// A spring of each node of the pair P towards the pair Q = (a.y, b.x) that
// straddles two column pairs: the differences are formed one component at a
// time, so Q is never assembled.
__device__ __forceinline__ float2 dstr(float ay, float bx, float2 p) { return make_float2(__fsub_rn(ay, p.x), __fsub_rn(bx, p.y)); }
__device__ __forceinline__ Vec2 spring2s(const Node2 &P, const Node2 &a, const Node2 &b, float2 ks, float2 kd,
                                         float L0)
{
    return spring2d(dstr(a.px.y, b.px.x, P.px), dstr(a.py.y, b.py.x, P.py), dstr(a.pz.y, b.pz.x, P.pz),
                    dstr(a.vx.y, b.vx.x, P.vx), dstr(a.vy.y, b.vy.x, P.vy), dstr(a.vz.y, b.vz.x, P.vz), ks, kd, L0);
}

// Sign bits set (node A in .x, node B in .y) where the segment from s to e
// lies on the far side of one face of the slab [lo, hi]: both ends below lo
// or both above hi.
__device__ __forceinline__ uint2 box_out_bits(float2 s, float2 e, float lo, float hi)
{
    const float2 a = sub2(s, bc(lo)), b = sub2(e, bc(lo)), c = sub2(bc(hi), s), d = sub2(bc(hi), e);
    return make_uint2((__float_as_uint(a.x) & __float_as_uint(b.x)) | (__float_as_uint(c.x) & __float_as_uint(d.x)),
                      (__float_as_uint(a.y) & __float_as_uint(b.y)) | (__float_as_uint(c.y) & __float_as_uint(d.y)));
}

// The wind's acceleration of a pair: amp * sin(a + b) with a the row's phase
// (time phase sinW, cosW plus the row's tr = (sin, cos)) and b the columns'.
// sin(a + b) = sin(a) cos(b) + cos(a) sin(b); every rounding is written out, so
// that every kernel gets the same bits.
__device__ __forceinline__ float2 wind_pair(float sinW, float cosW, float2 tr, float2 sinB, float2 cosB, float amp)
{
    const float sinR = __fmaf_rn(cosW, tr.x, __fmul_rn(sinW, tr.y));
    const float cosR = __fmaf_rn(cosW, tr.y, -__fmul_rn(sinW, tr.x));
    return mul2(bc(amp), fma2(bc(cosR), sinB, mul2(bc(sinR), cosB)));
}

// q - (ay, bx) for a pair q and the straddling pair (a.y, b.x), one
// component at a time.
__device__ __forceinline__ float2 rdstr(float2 q, float ay, float bx) { return make_float2(__fsub_rn(q.x, ay), __fsub_rn(q.y, bx)); }
// Kernel launch with the programmatic-serialisation attribute (see pdl_wait).
template <typename... KArgs, typename... Args>
cudaError_t launch_k(void (*kern)(KArgs...), int blocks, int threads, cudaStream_t s, Args &&...args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)blocks);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = 0;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = CLOTH_PDL;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, std::forward<Args>(args)...);
}
}  // namespace
