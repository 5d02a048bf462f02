// One substep of a small cloth as one kernel: springs, integration, collision.
//
// The column walk (cloth_step.cu) evaluates each spring once, but a warp
// takes three dependent row iterations for one row of output, and the collision
// pass is a second launch with its list in between.  A cloth that leaves the
// chip half empty is bound by that chain, not by arithmetic.  Here a thread
// owns two neighbouring nodes (a float2 pair, as in the walk), loads its
// twelve neighbours at once and evaluates all twelve springs, the six that end
// at it from the operands of their owners: twice the arithmetic, one round of
// loads and no exchange between lanes.  Forces are the same rounded operations
// on the same operands, summed in the walk's order, so the bits are the
// walk's.  A CTA owns 32 pairs; its W warps then go through the narrow phase of
// the nodes near the mesh, from shared memory, and the substep ends.
//
// Measured against the walk and the collision pass as two launches (graph
// replay, us per substep; n x n nodes lying on 20,480 triangles): n = 16
// 9.3 -> 6.2, 96 10.9 -> 6.7, 160 12.9 -> 8.2, 240 14.6 -> 11.5; without a mesh
// n = 16 3.7 -> 3.1, 64 to 160 4.1 -> 3.6, 240 4.6 -> 4.1, 330 5.7 -> 4.8.  What is
// left is the launch and one chain of loads per phase.
#include "cloth_collide.cuh"
#include "cloth_force.cuh"
#include "cloth_internal.h"

namespace {

// Loads that must follow the wait for the previous substep: the compiler may
// move a plain (or read-only) load across it, not these.
__device__ __forceinline__ float2 ld2(const float *p)
{
    float2 v;
    asm volatile("ld.global.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(p));
    return v;
}
__device__ __forceinline__ float ld1(const float *p)
{
    float v;
    asm volatile("ld.global.f32 %0, [%1];" : "=f"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ Node2 load_pair(const float *in, unsigned st, unsigned o)
{
    return {ld2(in + o), ld2(in + (o + st)), ld2(in + (o + 2u * st)), ld2(in + (o + 3u * st)), ld2(in + (o + 4u * st)),
            ld2(in + (o + 5u * st))};
}
struct Node1 {  // one node
    float px, py, pz, vx, vy, vz;
};
__device__ __forceinline__ Node1 load_one(const float *in, unsigned st, unsigned o)
{
    return {ld1(in + o), ld1(in + (o + st)), ld1(in + (o + 2u * st)), ld1(in + (o + 3u * st)), ld1(in + (o + 4u * st)),
            ld1(in + (o + 5u * st))};
}

// The spring forces of a pair, added up with the walk's rounding.  There the
// (+1,0) force is only ever added packed, and ptxas contracts that product and
// sum into one operation (for packed operands it does so in spite of the
// explicit rounding); the other forces travel through shuffles and are rounded
// before they are added.  Here both are written out: add_fused, and add_rounded
// with scalar products, which a packed sum cannot absorb.
struct Diff {  // far end minus owner, positions and velocities
    float2 dx, dy, dz, ux, uy, uz;
};
__device__ __forceinline__ Diff diff(const Node2 &P, const Node2 &Q)
{
    return {sub2(Q.px, P.px), sub2(Q.py, P.py), sub2(Q.pz, P.pz), sub2(Q.vx, P.vx), sub2(Q.vy, P.vy), sub2(Q.vz, P.vz)};
}
__device__ __forceinline__ float2 scale(const Diff &d, float2 ks, float2 kd, float L0)
{
    return spring_scale(d.dx, d.dy, d.dz, d.ux, d.uy, d.uz, ks, kd, L0);
}
__device__ __forceinline__ float2 prod(float2 a, float2 b) { return make_float2(__fmul_rn(a.x, b.x), __fmul_rn(a.y, b.y)); }
__device__ __forceinline__ Vec2 force(const Diff &d, float2 ks, float2 kd, float L0)
{
    const float2 s = scale(d, ks, kd, L0);
    return {prod(s, d.dx), prod(s, d.dy), prod(s, d.dz)};
}
__device__ __forceinline__ Vec2 add_rounded(Vec2 F, const Diff &d, float2 ks, float2 kd, float L0)
{
    return vadd(F, force(d, ks, kd, L0));
}
__device__ __forceinline__ Vec2 add_fused(Vec2 F, const Diff &d, float2 ks, float2 kd, float L0)
{
    const float2 s = scale(d, ks, kd, L0);
    return {fma2(s, d.dx, F.x), fma2(s, d.dy, F.y), fma2(s, d.dz, F.z)};
}
// Differences to and from a pair (a, b) that straddles two column pairs, a
// and b given per component.
__device__ __forceinline__ Diff to_pair(const Node2 &P, float apx, float bpx, float apy, float bpy, float apz,
                                        float bpz, float avx, float bvx, float avy, float bvy, float avz, float bvz)
{
    return {dstr(apx, bpx, P.px), dstr(apy, bpy, P.py), dstr(apz, bpz, P.pz), dstr(avx, bvx, P.vx),
            dstr(avy, bvy, P.vy), dstr(avz, bvz, P.vz)};
}
__device__ __forceinline__ Diff from_pair(const Node2 &Q, float apx, float bpx, float apy, float bpy, float apz,
                                          float bpz, float avx, float bvx, float avy, float bvy, float avz, float bvz)
{
    return {rdstr(Q.px, apx, bpx), rdstr(Q.py, apy, bpy), rdstr(Q.pz, apz, bpz), rdstr(Q.vx, avx, bvx),
            rdstr(Q.vy, avy, bvy), rdstr(Q.vz, avz, bvz)};
}
// the pair (b of the left pair, a of the right pair), and with one end a single node
#define STRADDLE(A, B) \
    (A).px.y, (B).px.x, (A).py.y, (B).py.x, (A).pz.y, (B).pz.x, (A).vx.y, (B).vx.x, (A).vy.y, (B).vy.x, (A).vz.y, (B).vz.x
#define ONE_PAIR(A, B) (A).px, (B).px.x, (A).py, (B).py.x, (A).pz, (B).pz.x, (A).vx, (B).vx.x, (A).vy, (B).vy.x, (A).vz, (B).vz.x
#define PAIR_ONE(A, B) (A).px.y, (B).px, (A).py.y, (B).py, (A).pz.y, (B).pz, (A).vx.y, (B).vx, (A).vy.y, (B).vy, (A).vz.y, (B).vz

// Constants of one direction's springs for the pair: per type, or per spring
// from the owners' slots at offsets oa (A's owner) and ob (B's); 0 where the
// spring does not exist (ea, eb; only looked at with EDGE: at the border).
template <bool PS, bool EDGE>
__device__ __forceinline__ void spring_consts(const StepParams &p, int dir, int type, long long oa, long long ob,
                                              bool ea, bool eb, float2 &ks, float2 &kd)
{
    if (PS) {
        const float *k = p.ks_slot + dir * p.stride, *d = p.kd_slot + dir * p.stride;
        ks = make_float2(!EDGE || ea ? __ldg(k + oa) : 0.0f, !EDGE || eb ? __ldg(k + ob) : 0.0f);
        kd = make_float2(!EDGE || ea ? __ldg(d + oa) : 0.0f, !EDGE || eb ? __ldg(d + ob) : 0.0f);
    } else {
        ks = make_float2(!EDGE || ea ? p.ks[type] : 0.0f, !EDGE || eb ? p.ks[type] : 0.0f);
        kd = make_float2(!EDGE || ea ? p.kd[type] : 0.0f, !EDGE || eb ? p.kd[type] : 0.0f);
    }
}

// Force on the pair (r, c), (r, c + 1) at offset o, own: the pair itself.
// EDGE: a neighbour may lie outside the grid (its loads are clamped into it and
// its springs get zero constants).
template <bool PS, bool EDGE>
__device__ __forceinline__ Vec2 pair_force(const StepParams &p, const float *in, int r, int c, const Node2 &own)
{
    const unsigned st = (unsigned)p.stride;
    const int ny = p.ny, nx = p.nx, pitch = p.pitch;
    auto at = [&](int rr, int cc) {  // offset of (rr, cc), clamped into the plane
        if (EDGE) {
            rr = min(max(rr, 0), ny - 1);
            cc = min(max(cc, 0), pitch - 1);
        }
        return (unsigned)rr * (unsigned)pitch + (unsigned)cc;
    };
    auto pair_at = [&](int rr, int cc) {  // cc even: the pair starting there
        if (EDGE) {
            rr = min(max(rr, 0), ny - 1);
            cc = min(max(cc, 0), pitch - 2);
        }
        return (unsigned)rr * (unsigned)pitch + (unsigned)cc;
    };
    const Node2 D2 = load_pair(in, st, pair_at(r + 2, c)), D1 = load_pair(in, st, pair_at(r + 1, c));
    const Node1 DR = load_one(in, st, at(r + 1, c + 2)), DL = load_one(in, st, at(r + 1, c - 1));
    const Node2 R = load_pair(in, st, pair_at(r, c + 2)), L = load_pair(in, st, pair_at(r, c - 2));
    const Node2 U2 = load_pair(in, st, pair_at(r - 2, c)), U1 = load_pair(in, st, pair_at(r - 1, c));
    const Node1 UL = load_one(in, st, at(r - 1, c - 1)), UR = load_one(in, st, at(r - 1, c + 2));
    const bool a1 = c + 1 < nx, a2 = c + 2 < nx, a3 = c + 3 < nx, l1 = c >= 1, l2 = c >= 2;
    const bool d1 = r + 1 < ny, d2 = r + 2 < ny, u1 = r >= 1, u2 = r >= 2;
    const long long o = (long long)r * pitch + c;
    float2 ks, kd;
    // owned springs, in the walk's order
    spring_consts<PS, EDGE>(p, 5, 2, o, o + 1, d2, d2, ks, kd);
    Vec2 F = force(diff(own, D2), ks, kd, p.L0[5]);
    spring_consts<PS, EDGE>(p, 1, 0, o, o + 1, d1, d1, ks, kd);
    F = add_fused(F, diff(own, D1), ks, kd, p.L0[1]);
    spring_consts<PS, EDGE>(p, 2, 1, o, o + 1, d1 && a1, d1 && a2, ks, kd);
    F = add_rounded(F, to_pair(own, PAIR_ONE(D1, DR)), ks, kd, p.L0[2]);
    spring_consts<PS, EDGE>(p, 3, 1, o, o + 1, d1 && l1, d1 && a1, ks, kd);
    F = add_rounded(F, to_pair(own, ONE_PAIR(DL, D1)), ks, kd, p.L0[3]);
    spring_consts<PS, EDGE>(p, 0, 0, o, o + 1, a1, a2, ks, kd);
    F = add_rounded(F, to_pair(own, STRADDLE(own, R)), ks, kd, p.L0[0]);
    spring_consts<PS, EDGE>(p, 4, 2, o, o + 1, a2, a3, ks, kd);
    F = add_rounded(F, diff(own, R), ks, kd, p.L0[4]);
    // springs that end here, their owners' forces
    spring_consts<PS, EDGE>(p, 5, 2, o - 2 * pitch, o - 2 * pitch + 1, u2, u2, ks, kd);
    Vec2 A = force(diff(U2, own), ks, kd, p.L0[5]);
    spring_consts<PS, EDGE>(p, 1, 0, o - pitch, o - pitch + 1, u1, u1, ks, kd);
    A = add_fused(A, diff(U1, own), ks, kd, p.L0[1]);
    spring_consts<PS, EDGE>(p, 2, 1, o - pitch - 1, o - pitch, u1 && l1, u1, ks, kd);
    A = add_rounded(A, from_pair(own, ONE_PAIR(UL, U1)), ks, kd, p.L0[2]);
    spring_consts<PS, EDGE>(p, 3, 1, o - pitch + 1, o - pitch + 2, u1 && a1, u1 && a2, ks, kd);
    A = add_rounded(A, from_pair(own, PAIR_ONE(U1, UR)), ks, kd, p.L0[3]);
    spring_consts<PS, EDGE>(p, 0, 0, o - 1, o, l1, true, ks, kd);
    Vec2 back = force(from_pair(own, STRADDLE(L, own)), ks, kd, p.L0[0]);
    spring_consts<PS, EDGE>(p, 4, 2, o - 2, o - 1, l2, l2, ks, kd);
    back = add_rounded(back, diff(L, own), ks, kd, p.L0[4]);
    return vsub(F, vadd(A, back));
}

// CTAs per SM up to which a cloth gets W warps per CTA, so that all are
// resident at once (registers); more lanes per node shorten its chain of loads.
// Two warps of 128 registers (8 CTAs per SM) beat listing the nodes for the
// collision pass on 256 x 256 and 272 x 272 nodes lying on the model, 12.9 against
// 15.5 us (11.8 now); in light contact, pulled over it, listing was ahead with 11.2
// against 12.3, until the narrow phase had more loads in flight (10.3).  Beyond
// that the nodes are listed, and from 12 CTAs per SM the walk takes over (its
// rows then have the warps they need).
#define CLOTH_NODE_W8 1
#define CLOTH_NODE_W4 3
#ifndef CLOTH_NODE_W2
#define CLOTH_NODE_W2 8
#endif
#define CLOTH_NODE_MAX 12

enum { NODE_FREE = 0, NODE_MESH = 1, NODE_EDGE = 2, NODE_LIST = 3 };

// MODE: no surface model; one, collided here; the edge narrow phase, whose
// kernels follow (cloth_step.cu); or a surface model whose nodes are listed
// for the collision pass that follows.  W warps per CTA: the first computes the
// CTA's 32 pairs, all of them collide.  REC: the adjoint's recompute.
//
// The CTA's nodes are the 64 plane positions from `base`.
template <int MODE, bool PS, bool REC, int W>
__device__ __forceinline__ void node_substep(const StepParams &p, const int par, const unsigned base)
{
    // per node of the CTA: start and end of the path, end velocity
    __shared__ float s_x[MODE == NODE_MESH ? 9 : 1][64];
    __shared__ int s_list[64], s_n;
    __shared__ unsigned s_stat[2];
    const int lane = threadIdx.x & 31;
    const unsigned st = (unsigned)p.stride;
    const float *in = par ? p.state1 : p.state0;
    float *out = par ? p.state0 : p.state1;
    float fs = 0.0f;
    if (threadIdx.x < 32) {
        const unsigned total = (unsigned)p.ny * (unsigned)p.pitch;
        unsigned o = base + 2u * (unsigned)lane;
        const bool active = o < total;
        if (!active) o = 0u;
        const int r = (int)(o / (unsigned)p.pitch), c = (int)(o - (unsigned)r * (unsigned)p.pitch);
        const bool okA = active && c < p.nx, okB = active && c + 1 < p.nx;
        // inputs that do not change from substep to substep
        unsigned pinw = 0u;
        if (p.pin_bits) pinw = __ldg(p.pin_bits + (o >> 5)) >> (o & 31u);
        float2 tr = make_float2(0.0f, 1.0f), tA = tr, tB = tr;
        if (p.has_wind) {
            tr = __ldg(p.wind_rows + r);
            if (c < p.nx) tA = __ldg(p.wind_cols + c);
            if (c + 1 < p.nx) tB = __ldg(p.wind_cols + c + 1);
        }
        pdl_wait();
        unsigned long long k = 0ull;
        if (p.has_wind || (blockIdx.x == 0 && lane == 0)) k = *(volatile unsigned long long *)&p.ctrl->kk[par];
        const Node2 own = load_pair(in, st, o);
        const bool inner = r >= 2 && r + 2 < p.ny && c >= 2 && c + 3 < p.nx;
        const Vec2 F = __all_sync(FULL, inner) ? pair_force<PS, false>(p, in, r, c, own)
                                               : pair_force<PS, true>(p, in, r, c, own);
        float2 ax = fma2(F.x, bc(p.inv_mass), bc(p.g[0]));
        float2 ay = fma2(F.y, bc(p.inv_mass), bc(p.g[1]));
        float2 az = fma2(F.z, bc(p.inv_mass), bc(p.g[2]));
        if (p.has_wind) {
            // sin(a + b) = sin(a) cos(b) + cos(a) sin(b), a = base + alpha_r
            float sinW, cosW;
            sincosf(wind_base(p.w_turn_step, p.w_turn0, k), &sinW, &cosW);
            const float2 w = wind_pair(sinW, cosW, tr, make_float2(tA.x, tB.x), make_float2(tA.y, tB.y), p.w_amp);
            ax = fma2(w, bc(p.w_dir[0]), ax);
            ay = fma2(w, bc(p.w_dir[1]), ay);
            az = fma2(w, bc(p.w_dir[2]), az);
        }
        const float2 dt = bc(p.dt);
        float2 wx = fma2(dt, ax, own.vx), wy = fma2(dt, ay, own.vy), wz = fma2(dt, az, own.vz);
        float2 xx = fma2(dt, wx, own.px), xy = fma2(dt, wy, own.py), xz = fma2(dt, wz, own.pz);
        if (pinw & 1u) {  // pinned nodes move kinematically: x += dt u, v = u (u = 0: fixed)
            xx.x = fmaf(p.dt, p.pin_vel[0], own.px.x); xy.x = fmaf(p.dt, p.pin_vel[1], own.py.x);
            xz.x = fmaf(p.dt, p.pin_vel[2], own.pz.x);
            wx.x = p.pin_vel[0]; wy.x = p.pin_vel[1]; wz.x = p.pin_vel[2];
        }
        if (pinw & 2u) {
            xx.y = fmaf(p.dt, p.pin_vel[0], own.px.y); xy.y = fmaf(p.dt, p.pin_vel[1], own.py.y);
            xz.y = fmaf(p.dt, p.pin_vel[2], own.pz.y);
            wx.y = p.pin_vel[0]; wy.y = p.pin_vel[1]; wz.y = p.pin_vel[2];
        }
        if (okA) {
            if (!okB) {  // B is padding: keep it zero
                xx.y = xy.y = xz.y = wx.y = wy.y = wz.y = 0.0f;
            }
            const float2 f2 = add2(add2(xx, xy), xz);
            fs = f2.x + f2.y;
            if (p.vstar) {  // velocity after integration, before the response (adjoint recompute)
                *(float2 *)(p.vstar + o) = wx;
                *(float2 *)(p.vstar + (o + st)) = wy;
                *(float2 *)(p.vstar + (o + 2u * st)) = wz;
            }
            *(float2 *)(out + o) = xx;
            *(float2 *)(out + (o + st)) = xy;
            *(float2 *)(out + (o + 2u * st)) = xz;
            *(float2 *)(out + (o + 3u * st)) = wx;
            *(float2 *)(out + (o + 4u * st)) = wy;
            *(float2 *)(out + (o + 5u * st)) = wz;
        }
        if (blockIdx.x == 0 && lane == 0) {
            // the other word is lower until this launch ends the substep
            if (*(volatile unsigned long long *)&p.ctrl->kk[par ^ 1] > k)
                atomicOr(&p.ctrl->flags, (unsigned)CTRL_FLAG_PARITY);
            if (MODE == NODE_EDGE || MODE == NODE_LIST) p.ctrl->kc = k;
            else ctrl_end_k(p.ctrl, k);
        }
        if (MODE == NODE_MESH || MODE == NODE_LIST) {
            // the nodes whose path box reaches the mesh's padded vertex box (as in the walk)
            const bool needA = okA && !(pinw & 1u) && fmaxf(own.px.x, xx.x) >= p.mlo[0] &&
                               fminf(own.px.x, xx.x) <= p.mhi[0] && fmaxf(own.py.x, xy.x) >= p.mlo[1] &&
                               fminf(own.py.x, xy.x) <= p.mhi[1] && fmaxf(own.pz.x, xz.x) >= p.mlo[2] &&
                               fminf(own.pz.x, xz.x) <= p.mhi[2];
            const bool needB = okB && !(pinw & 2u) && fmaxf(own.px.y, xx.y) >= p.mlo[0] &&
                               fminf(own.px.y, xx.y) <= p.mhi[0] && fmaxf(own.py.y, xy.y) >= p.mlo[1] &&
                               fminf(own.py.y, xy.y) <= p.mhi[1] && fmaxf(own.pz.y, xz.y) >= p.mlo[2] &&
                               fminf(own.pz.y, xz.y) <= p.mhi[2];
            const unsigned mA = __ballot_sync(FULL, needA), mB = __ballot_sync(FULL, needB);
            const unsigned lt = (1u << lane) - 1u;
            const int at = __popc(mA & lt) + __popc(mB & lt);
            if (MODE == NODE_LIST) {
                if (mA | mB) {
                    unsigned w = 0u;
                    if (lane == 0) w = atomicAdd(p.coll_count + par, (unsigned)(__popc(mA) + __popc(mB)));
                    w = __shfl_sync(FULL, w, 0) + (unsigned)at;
                    if (needA) p.coll_list[w] = (int)o;
                    if (needB) p.coll_list[w + needA] = (int)o + 1;
                }
            } else {
                if (needA) s_list[at] = 2 * lane;
                if (needB) s_list[at + needA] = 2 * lane + 1;
                auto put = [&](int q, float2 v) { *(float2 *)&s_x[q][2 * lane] = v; };
                put(0, own.px); put(1, own.py); put(2, own.pz);
                put(3, xx); put(4, xy); put(5, xz);
                put(6, wx); put(7, wy); put(8, wz);
                if (lane == 0) {
                    s_n = __popc(mA) + __popc(mB);
                    s_stat[0] = s_stat[1] = 0u;
                }
            }
        }
    }
    if (MODE == NODE_MESH) {
        if (W == 1) __syncwarp();
        else __syncthreads();
        const int n = s_n;
        if (n > 0) {
            unsigned ntest = 0u, nhit = 0u;
            auto pass = [&](auto group) {
                constexpr int G = decltype(group)::value;
                for (int i0 = 0; i0 < n; i0 += 32 * W / G) {
                    const int i = i0 + (int)threadIdx.x / G;
                    const bool valid = i < n;
                    const int j = valid ? s_list[i] : 0;
                    const unsigned o = base + (unsigned)j;
                    float3 x;
                    if (collide_path<REC, G, true>(OneCloth{p}, 0, p, valid, s_x[0][j], s_x[1][j], s_x[2][j], s_x[3][j],
                                             s_x[4][j], s_x[5][j], (long long)o, x, ntest)) {
                        out[o] = x.x;
                        out[o + st] = x.y;
                        out[o + 2u * st] = x.z;
                        out[o + 3u * st] = s_x[6][j] * p.restitution;
                        out[o + 4u * st] = s_x[7][j] * p.restitution;
                        out[o + 5u * st] = s_x[8][j] * p.restitution;
                        fs += x.x + x.y + x.z;
                        nhit++;
                    }
                }
            };
            if (8 * n <= 32 * W) pass(std::integral_constant<int, 8>());
            else pass(std::integral_constant<int, W == 1 ? 1 : W / 2>());
            const unsigned h = __reduce_add_sync(FULL, nhit), t = __reduce_add_sync(FULL, ntest);
            if (W == 1) {
                if (lane == 0) coll_stats_store(p.ctrl, (unsigned)n, t, h);
            } else {
                if (lane == 0) {
                    if (t) atomicAdd(&s_stat[0], t);
                    if (h) atomicAdd(&s_stat[1], h);
                }
                __syncthreads();
                if (threadIdx.x == 0) coll_stats_store(p.ctrl, (unsigned)n, s_stat[0], s_stat[1]);
            }
        }
    }
    if (__any_sync(FULL, !isfinite(fs)) && lane == 0) atomicOr(&p.ctrl->flags, (unsigned)CTRL_FLAG_NONFINITE);
}

constexpr int node_min_ctas(int W) { return W == 1 ? CLOTH_NODE_MAX : W == 2 ? CLOTH_NODE_W2 : W == 4 ? CLOTH_NODE_W4 : CLOTH_NODE_W8; }

template <int MODE, bool PS, bool REC, int W>
__global__ void __launch_bounds__(32 * W, node_min_ctas(W)) node_kernel(const __grid_constant__ StepParams p)
{
    pdl_launch_dependents();
    node_substep<MODE, PS, REC, W>(p, p.parity & 1, 64u * blockIdx.x);
}

// A batch of small cloths: a CTA per (cloth, 64 positions) of the list b.groups.
template <int MODE, bool PS, int W>
__global__ void __launch_bounds__(32 * W, node_min_ctas(W)) node_batch_kernel(const __grid_constant__ BatchArgs b)
{
    __shared__ StepParams p;
    pdl_launch_dependents();
    const int2 g = __ldg(b.groups + blockIdx.x);
    const unsigned *src = (const unsigned *)(b.params + g.x);  // does not change from substep to substep
    for (int w = threadIdx.x; w < (int)(sizeof(StepParams) / 4); w += 32 * W) ((unsigned *)&p)[w] = __ldg(src + w);
    if (W == 1) __syncwarp();
    else __syncthreads();
    node_substep<MODE, PS, false, W>(p, b.parity & 1, 64u * (unsigned)g.y);
}

template <int MODE, int W>
cudaError_t launch_batch_mode(const BatchArgs &b, cudaStream_t s)
{
    return b.variant & BATCH_VAR_PER_SPRING ? launch_k(node_batch_kernel<MODE, true, W>, b.n_groups, 32 * W, s, b)
                                            : launch_k(node_batch_kernel<MODE, false, W>, b.n_groups, 32 * W, s, b);
}

template <int MODE, int W>
cudaError_t launch_mode(const StepParams &p, int blocks, cudaStream_t s)
{
    if (MODE == NODE_MESH && p.cdata) return launch_k(node_kernel<MODE, true, MODE == NODE_MESH, W>, blocks, 32 * W, s, p);
    return p.ks_slot ? launch_k(node_kernel<MODE, true, false, W>, blocks, 32 * W, s, p)
                     : launch_k(node_kernel<MODE, false, false, W>, blocks, 32 * W, s, p);
}

int node_ctas(const StepParams &p) { return (int)(((long long)p.ny * p.pitch + 63) / 64); }

}  // namespace

bool node_kernel_fits(const StepParams &p)
{
    return !p.force && !(p.cdata && node_ctas(p) > CLOTH_NODE_W2 * p.sms) && node_ctas(p) <= CLOTH_NODE_MAX * p.sms;
}

cudaError_t launch_node_substep(const StepParams &p, cudaStream_t s)
{
    const int blocks = node_ctas(p);
    if (!p.has_mesh) return launch_mode<NODE_FREE, 1>(p, blocks, s);
    if (p.edge_resp) {
        const cudaError_t e = launch_mode<NODE_EDGE, 1>(p, blocks, s);
        return e == cudaSuccess ? launch_collide(p, s) : e;
    }
    if (blocks <= CLOTH_NODE_W8 * p.sms) return launch_mode<NODE_MESH, 8>(p, blocks, s);
    if (blocks <= CLOTH_NODE_W4 * p.sms) return launch_mode<NODE_MESH, 4>(p, blocks, s);
    if (blocks <= CLOTH_NODE_W2 * p.sms) return launch_mode<NODE_MESH, 2>(p, blocks, s);
    const cudaError_t e = launch_mode<NODE_LIST, 1>(p, blocks, s);
    return e == cudaSuccess ? launch_collide(p, s) : e;
}

// As for one cloth, by the batch's number of groups; a batch that mixes walk
// variants or has more groups than are resident takes the persistent walk.
bool node_batch_fits(long long groups, int variant, int sms)
{
    return variant != BATCH_VAR_MIXED && groups <= (long long)(variant & BATCH_VAR_MESH ? CLOTH_NODE_W2 : CLOTH_NODE_MAX) * sms;
}

cudaError_t launch_node_batch(const BatchArgs &b, cudaStream_t s)
{
    if (!(b.variant & BATCH_VAR_MESH)) return launch_batch_mode<NODE_FREE, 1>(b, s);
    if (b.n_groups <= CLOTH_NODE_W8 * b.sms) return launch_batch_mode<NODE_MESH, 8>(b, s);
    if (b.n_groups <= CLOTH_NODE_W4 * b.sms) return launch_batch_mode<NODE_MESH, 4>(b, s);
    return launch_batch_mode<NODE_MESH, 2>(b, s);
}
