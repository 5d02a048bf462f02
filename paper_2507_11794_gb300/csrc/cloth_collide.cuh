// Collision of a node's substep path with the surface model (device code
// shared by the stepping kernels and the adjoint's recompute).
//
// Broad phase (not in the paper, which tests every pair; a uniform grid over
// the surface triangles): the path S -> E is boxed and the triangles listed in
// the grid cells of that box are the candidates; a triangle listed in several
// of those cells is tested only in the first cell the two boxes share.
// Narrow phase: the extended Moller-Trumbore test of Section 3 on the path
// against each candidate.  Response (Algorithm 2): with K hits at
// distances t_k along r = (E - S)/|E - S|, the node moves to
// S + mean_k max(t_k - delta, 0) r and its velocity is scaled by the
// restitution factor.
#pragma once

#include "cloth_internal.h"

// Path of one node: start S, unit direction r, length L.
struct CollPath {
    float sx, sy, sz, rx, ry, rz, L;
};

// Grid-cell box of a path (cell_coord on both ends, per axis).
struct CollBox {
    int lox, loy, loz, hix, hiy, hiz;
};

__device__ __forceinline__ CollBox coll_box(const StepParams &p, float sx, float sy, float sz, float ex, float ey,
                                            float ez)
{
    CollBox b;
    b.lox = cell_coord(fminf(sx, ex), p.go[0], p.ginv, p.gd[0]);
    b.hix = cell_coord(fmaxf(sx, ex), p.go[0], p.ginv, p.gd[0]);
    b.loy = cell_coord(fminf(sy, ey), p.go[1], p.ginv, p.gd[1]);
    b.hiy = cell_coord(fmaxf(sy, ey), p.go[1], p.ginv, p.gd[1]);
    b.loz = cell_coord(fminf(sz, ez), p.go[2], p.ginv, p.gd[2]);
    b.hiz = cell_coord(fmaxf(sz, ez), p.go[2], p.ginv, p.gd[2]);
    return b;
}

// a b - c d and a b + c d + e f with every rounding written out: what the
// compiler contracts differs from kernel to kernel, and a node's response has to
// come out the same in all of them.
__device__ __forceinline__ float det_rn(float a, float b, float c, float d) { return __fmaf_rn(a, b, -__fmul_rn(c, d)); }
__device__ __forceinline__ float dot_rn(float a, float b, float c, float d, float e, float f)
{
    return __fmaf_rn(e, f, __fmaf_rn(a, b, __fmul_rn(c, d)));
}

// One candidate: triangle record (A, B, C) = (v0, e1, e2) met in cell
// (cx, cy, cz) of a box whose low corner is (lox, loy, loz).  Returns true on a
// hit, with th the distance along r, over = th - delta (of the rounded th,
// whichever lane adds it up) and f = 1/a (a = e1 . (r x e2)).
__device__ __forceinline__ bool coll_test(const StepParams &p, const CollPath &q, const float4 &A, const float4 &B,
                                          const float4 &C, int cx, int cy, int cz, int lox, int loy, int loz, float &th,
                                          float &over, float &f)
{
    // the record's w lanes hold the low cell of the triangle's box
    if (max(__float_as_int(A.w), lox) != cx || max(__float_as_int(B.w), loy) != cy ||
        max(__float_as_int(C.w), loz) != cz)
        return false;
    // extended Moller-Trumbore: edge S -> E, direction r, length L
    const float hx = det_rn(q.ry, C.z, q.rz, C.y);
    const float hy = det_rn(q.rz, C.x, q.rx, C.z);
    const float hz = det_rn(q.rx, C.y, q.ry, C.x);
    const float a = dot_rn(B.x, hx, B.y, hy, B.z, hz);
    if (fabsf(a) < p.eps) return false;
    f = 1.0f / a;
    const float qx0 = __fsub_rn(q.sx, A.x), qy0 = __fsub_rn(q.sy, A.y), qz0 = __fsub_rn(q.sz, A.z);
    const float u = __fmul_rn(f, dot_rn(qx0, hx, qy0, hy, qz0, hz));
    if (u < 0.0f || u > 1.0f) return false;
    const float qx = det_rn(qy0, B.z, qz0, B.y);
    const float qy = det_rn(qz0, B.x, qx0, B.z);
    const float qz = det_rn(qx0, B.y, qy0, B.x);
    const float v = __fmul_rn(f, dot_rn(q.rx, qx, q.ry, qy, q.rz, qz));
    th = __fmul_rn(f, dot_rn(C.x, qx, C.y, qy, C.z, qz));
    over = __fsub_rn(th, p.delta);
    if (v < 0.0f || u + v > 1.0f) return false;
    return th > p.tmin && th < q.L;
}

// The same for grid entry e; A, B, C receive its record.
__device__ __forceinline__ bool coll_candidate(const StepParams &p, const CollPath &q, long long e, int cx, int cy,
                                               int cz, int lox, int loy, int loz, float &th, float &over, float &f,
                                               float4 &A, float4 &B, float4 &C)
{
    A = __ldg(p.etri + 3 * e);
    B = __ldg(p.etri + 3 * e + 1);
    C = __ldg(p.etri + 3 * e + 2);
    return coll_test(p, q, A, B, C, cx, cy, cz, lox, loy, loz, th, over, f);
}

// Point S + th r of a path, each coordinate one rounded fused multiply-add,
// so every kernel that computes a hit point gets the same bits.
__device__ __forceinline__ float3 coll_hit_point(const CollPath &q, float th)
{
    return make_float3(__fmaf_rn(th, q.rx, q.sx), __fmaf_rn(th, q.ry, q.sy), __fmaf_rn(th, q.rz, q.sz));
}

// Path of S -> E; false when it is shorter than eps (no test).
__device__ __forceinline__ bool coll_path(const StepParams &p, float sx, float sy, float sz, float ex, float ey,
                                          float ez, CollPath &q)
{
    const float dx = __fsub_rn(ex, sx), dy = __fsub_rn(ey, sy), dz = __fsub_rn(ez, sz);
    q.L = sqrtf(dot_rn(dx, dx, dy, dy, dz, dz));
    if (!(q.L >= p.eps)) return false;
    q.sx = sx; q.sy = sy; q.sz = sz;
    q.rx = dx / q.L; q.ry = dy / q.L; q.rz = dz / q.L;
    return true;
}

struct OneCloth {  // coll_cells' source of parameters for one cloth
    const StepParams &p;
    __device__ const StepParams &params(int) const { return p; }
};

// Candidate filter: every grid entry carries its triangle's box in units of
// 1 / 64 of a cell (coarser on long grids, see grid_filter_scale; grown by one
// unit and the rounding of the mesh's coordinates), laid out so
// that three subtractions compare it with a path's box on all six sides: word
// lanes of 15 bits under a guard bit, T = (hx, hy) (hz, M - lx) (M - ly,
// M - lz) for the triangle and N = (lo x, lo y) (lo z, M - hi x) (...) for the
// path, M = 32767; the boxes overlap iff every lane of T is >= that of N, i.e.
// iff no guard bit is borrowed from.  A path can only hit a triangle whose
// box it overlaps, so the test below it runs on the entries that pass.  The
// float32 test by itself can also accept a triangle far outside whose box the
// path lies, in the triangle's own plane: its errors in u, v and t grow as 1 / a,
// and a path along a large tilted triangle has a far below the triangle's size.
// The filter turns those away; whatever looks at hits has to look through it.
// The fourth word has bit a (0, 1, 2) where the entry's cell is the first of
// the triangle's box along axis a: a triangle listed in several cells of a
// path's box is tested only in the first cell the two boxes share, which is
// this one iff along every axis the cell is the path box's first or that bit
// is set (the same rule coll_candidate applies to the full record).
struct CollWords {
    unsigned a, b, c;
};

__device__ __forceinline__ CollWords coll_words(const StepParams &p, float sx, float sy, float sz, float ex, float ey,
                                                float ez, const CollPath &q)
{
    if (p.tmin < 0.0f) {  // hits behind the start count: the box reaches back to S + tmin r
        sx = fmaf(p.tmin, q.rx, sx);
        sy = fmaf(p.tmin, q.ry, sy);
        sz = fmaf(p.tmin, q.rz, sz);
    }
    const unsigned lx = grid_filter_coord(fminf(sx, ex), p.go[0], p.qs), hx = grid_filter_coord(fmaxf(sx, ex), p.go[0], p.qs);
    const unsigned ly = grid_filter_coord(fminf(sy, ey), p.go[1], p.qs), hy = grid_filter_coord(fmaxf(sy, ey), p.go[1], p.qs);
    const unsigned lz = grid_filter_coord(fminf(sz, ez), p.go[2], p.qs), hz = grid_filter_coord(fmaxf(sz, ez), p.go[2], p.qs);
    return {lx | ly << 16, lz | (GRID_FILTER_MAX - hx) << 16, (GRID_FILTER_MAX - hy) | (GRID_FILTER_MAX - hz) << 16};
}
// need: bit a set where the cell is not the path box's first along axis a.
__device__ __forceinline__ bool coll_overlap(const uint4 &t, const CollWords &n, unsigned need)
{
    return (((t.x - n.a) & (t.y - n.b) & (t.z - n.c)) & GRID_FILTER_GUARD) == GRID_FILTER_GUARD && !(need & ~t.w);
}
__device__ __forceinline__ unsigned coll_need(const CollBox &bx, int cx, int cy, int cz)
{
    return (cx != bx.lox) | (cy != bx.loy) << 1 | (cz != bx.loz) << 2;
}

__device__ __forceinline__ float coll_shfl(float v, int src) { return __shfl_sync(0xffffffffu, v, src); }

// What a path's hits are added to.  add<G>: every lane of a group of G brings
// one tested candidate (hit: whether it hit; th, over, f, B, C as from
// coll_candidate) and the group adds the hits in lane order, all of its lanes
// ending with the same sums; converged warps only for G > 1.  from(l): lane
// l's, in every lane.
//
// A node's: K and sum max(t - delta, 0) and, for the adjoint's recompute (REC),
// over the active hits (t > delta) g1 = sum n/a and g2 = sum t n/a (n = e1 x e2),
// the derivatives of t w.r.t. S and r.
template <bool REC>
struct NodeHits {
    int K;
    float acc, g1[REC ? 3 : 1], g2[REC ? 3 : 1];

    __device__ __forceinline__ void one(float val, float th, float f, const float4 &B, const float4 &C)
    {
        K++;
        acc += val;
        if constexpr (REC) {
            if (val > 0.0f) {
                const float nx = det_rn(B.y, C.z, B.z, C.y), ny = det_rn(B.z, C.x, B.x, C.z), nz = det_rn(B.x, C.y, B.y, C.x);
                // products rounded before they are added
                g1[0] = __fadd_rn(g1[0], __fmul_rn(nx, f));
                g1[1] = __fadd_rn(g1[1], __fmul_rn(ny, f));
                g1[2] = __fadd_rn(g1[2], __fmul_rn(nz, f));
                g2[0] = __fadd_rn(g2[0], __fmul_rn(__fmul_rn(th, nx), f));
                g2[1] = __fadd_rn(g2[1], __fmul_rn(__fmul_rn(th, ny), f));
                g2[2] = __fadd_rn(g2[2], __fmul_rn(__fmul_rn(th, nz), f));
            }
        }
    }
    template <int G>
    __device__ __forceinline__ void add(const StepParams &, const CollPath &, bool hit, float th, float over, float f,
                                        const float4 &B, const float4 &C)
    {
        const float val = fmaxf(over, 0.0f);
        if constexpr (G == 1) {
            if (hit) one(val, th, f, B, C);
        } else {
            const int lane = threadIdx.x & 31, gbase = lane & ~(G - 1);
            unsigned hm = (__ballot_sync(0xffffffffu, hit) >> gbase) & (0xffffffffu >> (32 - G));
            while (__any_sync(0xffffffffu, hm != 0u)) {
                const int src = hm ? gbase + __ffs((int)hm) - 1 : lane;
                const float hv = coll_shfl(val, src);
                float ht = 0.0f, hf = 0.0f;
                float4 hB = B, hC = C;
                if constexpr (REC) {
                    ht = coll_shfl(th, src);
                    hf = coll_shfl(f, src);
                    hB.x = coll_shfl(B.x, src); hB.y = coll_shfl(B.y, src); hB.z = coll_shfl(B.z, src);
                    hC.x = coll_shfl(C.x, src); hC.y = coll_shfl(C.y, src); hC.z = coll_shfl(C.z, src);
                }
                if (hm) one(hv, ht, hf, hB, hC);
                hm &= hm - 1u;
            }
        }
    }
    __device__ __forceinline__ NodeHits from(int l) const
    {
        NodeHits t;
        t.K = __shfl_sync(0xffffffffu, K, l);
        t.acc = coll_shfl(acc, l);
#pragma unroll
        for (int a = 0; a < (REC ? 3 : 1); a++) {
            t.g1[a] = REC ? coll_shfl(g1[a], l) : 0.0f;
            t.g2[a] = REC ? coll_shfl(g2[a], l) : 0.0f;
        }
        return t;
    }
};

// ------------------------------------------------------------ list pass
// The walk appends the nodes whose path box meets the box of the mesh's
// vertices.  A lane (or a group of lanes, see collide_list) per listed node: it
// boxes the path and goes through its cells (mostly one) in x, y, z order.
// Per cell it first runs the filter over up to 32 entries and keeps the
// survivors as a bit mask (16 B and a handful of instructions per entry,
// neighbouring lanes reading the same lines), then tests the survivors (a few
// per node near the surface, 48 B and the full test each), all lanes of the
// warp together.  Hits are added in candidate order,
// so the sum does not depend on how the work is spread.  What is long is
// walked by the whole warp: a path of more than COLL_MAXC cells, and a cell
// of more than COLL_MAXE entries, 32 candidates at a time.
constexpr int COLL_WARPS = 8;  // warps per CTA of the collision kernels
constexpr int COLL_MAXC = 8;   // cells of a box one lane goes through
constexpr int COLL_MAXE = 96;  // entries of a cell one lane goes through

// Records the response data of a hit node at plane offset o for the reverse
// pass: m, r, g1 / K, g2 / K (the factors it multiplies by the adjoints) and
// the node's bit.
__device__ __forceinline__ void coll_record(const StepParams &p, long long o, float m, float K, float rx, float ry,
                                            float rz, const float g1[3], const float g2[3])
{
    const long long st = p.stride;
    const float invK = 1.0f / K;
    float *cd = p.cdata;
    cd[o] = m;
    cd[st + o] = rx;
    cd[2 * st + o] = ry;
    cd[3 * st + o] = rz;
    cd[4 * st + o] = g1[0] * invK;
    cd[5 * st + o] = g1[1] * invK;
    cd[6 * st + o] = g1[2] * invK;
    cd[7 * st + o] = g2[0] * invK;
    cd[8 * st + o] = g2[1] * invK;
    cd[9 * st + o] = g2[2] * invK;
    atomicOr(p.cbits + (o >> 5), 1u << (o & 31));
}

// 32 candidates of one path tested by the warp, one per lane (have: whether
// the lane has one, entry e of cell (cx, cy, cz)).  Every lane passes the same
// path and ends with the same sums.
template <class Hits>
__device__ __forceinline__ void coll_warp_round(const StepParams &p, const CollPath &q, const CollWords &w,
                                                const CollBox &bx, bool have, long long e, int cx, int cy, int cz,
                                                Hits &s)
{
    float th = 0.0f, over = 0.0f, f = 0.0f;
    float4 A, B = make_float4(0.0f, 0.0f, 0.0f, 0.0f), C = B;
    const bool hit = have && coll_overlap(__ldg(p.efil + e), w, coll_need(bx, cx, cy, cz)) &&
                     coll_candidate(p, q, e, cx, cy, cz, bx.lox, bx.loy, bx.loz, th, over, f, A, B, C);
    s.template add<32>(p, q, hit, th, over, f, B, C);
}

// All cells of a long path walked by the whole warp (every lane passes the
// same arguments): 32 cells at a time, x fastest, then their candidates 32 at
// a time in cell order, so the hits come in the order of a walk by one thread.
// Returns the number of candidates.
template <class Hits>
__device__ __noinline__ unsigned coll_wide(const StepParams &p, const CollPath q, const CollWords w, const CollBox bx,
                                           Hits &s)
{
    const int lane = threadIdx.x & 31;
    const int nxc = bx.hix - bx.lox + 1, nyc = bx.hiy - bx.loy + 1, nzc = bx.hiz - bx.loz + 1;
    const long long nxy = (long long)nxc * nyc, ncell = nxy * nzc;
    unsigned tested = 0u;
    for (long long c0 = 0; c0 < ncell; c0 += 32) {
        const long long cc = c0 + lane;
        int e0 = 0, cnt = 0, cx = 0, cy = 0, cz = 0;
        if (cc < ncell) {
            cz = bx.loz + (int)(cc / nxy);
            const int rem = (int)(cc - (long long)(cz - bx.loz) * nxy);
            cy = bx.loy + rem / nxc;
            cx = bx.lox + rem % nxc;
            const long long cell = ((long long)cz * p.gd[1] + cy) * p.gd[0] + cx;
            e0 = __ldg(p.cell_start + cell);
            cnt = __ldg(p.cell_start + cell + 1) - e0;
        }
        int incl = cnt;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, incl, d);
            if (lane >= d) incl += t;
        }
        const int total = __shfl_sync(0xffffffffu, incl, 31);
        const int excl = incl - cnt;
        tested += (unsigned)total;
        for (int r0 = 0; r0 < total; r0 += 32) {
            const int j = r0 + lane;
            // the lane whose cell holds candidate j: the last with excl <= j
            int ow = 0;
#pragma unroll
            for (int step = 16; step > 0; step >>= 1)
                if (__shfl_sync(0xffffffffu, excl, ow + step) <= j) ow += step;
            const int oe0 = __shfl_sync(0xffffffffu, e0, ow), oex = __shfl_sync(0xffffffffu, excl, ow);
            const int ocx = __shfl_sync(0xffffffffu, cx, ow), ocy = __shfl_sync(0xffffffffu, cy, ow),
                      ocz = __shfl_sync(0xffffffffu, cz, ow);
            coll_warp_round(p, q, w, bx, j < total, (long long)oe0 + (j - oex), ocx, ocy, ocz, s);
        }
    }
    return tested;
}

// Where the entries of a cell start and end.
__device__ __forceinline__ int2 coll_run(const StepParams &p, int cx, int cy, int cz)
{
    const int *c = p.cell_start + ((long long)cz * p.gd[1] + cy) * p.gd[0] + cx;
    return make_int2(__ldg(c), __ldg(c + 1));
}

// The hits of every lane's path (ncell cells of its box; 0: none), G lanes per
// path: the lanes of a group are neighbours in the warp, bring the same path
// and end with the same sums.  wide: the path has more than the caller's limit of
// cells (ncell = 0) and is walked by the whole warp; its candidates are counted
// with COUNT_WIDE.  src.params(cloth) are the path's parameters.  ntest
// accumulates, in a group's first lane, the candidates.
//
// A lane's time is a chain of loads: of 17 filter words in a cell, four at a time
// and the last one alone, 3,100 cycles, then 1,400 per survivor (256 x 256 nodes
// pulled over 81,920 triangles, one lane per node; twice that from DRAM).  DEEP,
// for kernels with the registers for it, takes the first cell's entries (run) from
// the caller, who can load them ahead, and has up to eight filter words in flight,
// past the end the last one again, and with one lane per path the next survivor's
// record.
template <int G, bool COUNT_WIDE, bool DEEP, class Src, class Hits>
__device__ __forceinline__ void coll_cells(const Src &src, int cloth, const StepParams &p, const CollPath &q,
                                           const CollBox &bx, const CollWords &w, int2 run, int ncell, bool wide,
                                           Hits &s, unsigned &ntest)
{
    constexpr unsigned FULLW = 0xffffffffu;
    const int lane = threadIdx.x & 31, sub = lane % G, gbase = lane - sub;
    const int ncw = __reduce_max_sync(FULLW, ncell);
    int cx = bx.lox, cy = bx.loy, cz = bx.loz;
    for (int c = 0; c < ncw; c++) {
        int e0 = 0, cnt = 0;
        if (c < ncell) {
            if (c > 0 || !DEEP) run = coll_run(p, cx, cy, cz);
            e0 = run.x;
            cnt = run.y - e0;
            if (sub == 0) ntest += (unsigned)cnt;
        }
        const unsigned need = coll_need(bx, cx, cy, cz);
        const bool big = cnt > COLL_MAXE;
        const int own = big ? 0 : cnt;
        for (int b = 0; __any_sync(FULLW, b < own); b += 32) {
            const int n = min(own - b, 32);
            unsigned m = 0u;  // the entries of this run that pass the filter
            const uint4 *fil = p.efil + e0 + b;
            if constexpr (DEEP) {
                constexpr int U = G > 4 ? 32 / G : 8;  // words in flight
                for (int t = sub; t < n; t += U * G) {
                    uint4 f[U];
#pragma unroll
                    for (int j = 0; j < U; j++) f[j] = __ldg(fil + min(t + j * G, n - 1));
#pragma unroll
                    for (int j = 0; j < U; j++) m |= (unsigned)coll_overlap(f[j], w, need) << ((t + j * G) & 31);
                }
                if (n > 0) m &= 0xffffffffu >> (32 - n);
                else m = 0u;
            } else {
#pragma unroll 4
                for (int t = sub; t < n; t += G) m |= (unsigned)coll_overlap(__ldg(fil + t), w, need) << t;
            }
#pragma unroll
            for (int d = 1; d < G; d <<= 1) m |= __shfl_xor_sync(FULLW, m, d);
            if constexpr (DEEP && G == 1) {
                float4 nA, nB, nC;  // the next survivor's record
                int t = __ffs((int)m) - 1;
                auto fetch = [&]() {
                    const float4 *r = p.etri + 3 * ((long long)e0 + b + t);
                    nA = __ldg(r); nB = __ldg(r + 1); nC = __ldg(r + 2);
                };
                if (t >= 0) fetch();
                while (__any_sync(FULLW, t >= 0)) {
                    if (t >= 0) {
                        const float4 A = nA, B = nB, C = nC;
                        m &= m - 1u;
                        t = __ffs((int)m) - 1;
                        if (t >= 0) fetch();
                        float th, over, f;
                        const bool hit = coll_test(p, q, A, B, C, cx, cy, cz, bx.lox, bx.loy, bx.loz, th, over, f);
                        s.template add<1>(p, q, hit, th, over, f, B, C);
                    }
                }
            }
            while (__any_sync(FULLW, m != 0u)) {
                // the group's next G survivors, one per lane in entry order
                unsigned mine = m;
#pragma unroll
                for (int t = 0; t < G; t++) {
                    if (t < sub) mine &= mine - 1u;
                    m &= m - 1u;
                }
                const int t = __ffs((int)mine) - 1;
                float th = 0.0f, over = 0.0f, f = 0.0f;
                float4 A, B = make_float4(0.0f, 0.0f, 0.0f, 0.0f), C = B;
                const bool hit = t >= 0 && coll_candidate(p, q, (long long)e0 + b + t, cx, cy, cz, bx.lox, bx.loy,
                                                          bx.loz, th, over, f, A, B, C);
                s.template add<G>(p, q, hit, th, over, f, B, C);
            }
        }
        // crowded cells, one path's at a time over the whole warp
        for (unsigned bm = __ballot_sync(FULLW, big && sub == 0); bm; bm &= bm - 1u) {
            const int l = __ffs((int)bm) - 1;
            const CollPath lq = {coll_shfl(q.sx, l), coll_shfl(q.sy, l), coll_shfl(q.sz, l), coll_shfl(q.rx, l),
                                 coll_shfl(q.ry, l), coll_shfl(q.rz, l), coll_shfl(q.L, l)};
            const CollWords lw = {__shfl_sync(FULLW, w.a, l), __shfl_sync(FULLW, w.b, l), __shfl_sync(FULLW, w.c, l)};
            CollBox lb = bx;
            lb.lox = __shfl_sync(FULLW, bx.lox, l);
            lb.loy = __shfl_sync(FULLW, bx.loy, l);
            lb.loz = __shfl_sync(FULLW, bx.loz, l);
            const int le0 = __shfl_sync(FULLW, e0, l), lcnt = __shfl_sync(FULLW, cnt, l);
            const int lcx = __shfl_sync(FULLW, cx, l), lcy = __shfl_sync(FULLW, cy, l), lcz = __shfl_sync(FULLW, cz, l);
            const StepParams &lp = src.params(__shfl_sync(FULLW, cloth, l));
            Hits t = s.from(l);
            for (int r0 = 0; r0 < lcnt; r0 += 32)
                coll_warp_round(lp, lq, lw, lb, r0 + lane < lcnt, (long long)le0 + r0 + lane, lcx, lcy, lcz, t);
            if (gbase == l) s = t;
        }
        if (++cx > bx.hix) {
            cx = bx.lox;
            if (++cy > bx.hiy) {
                cy = bx.loy;
                cz++;
            }
        }
    }
    // long paths, one at a time over the whole warp
    for (unsigned wm = __ballot_sync(FULLW, wide && sub == 0); wm; wm &= wm - 1u) {
        const int l = __ffs((int)wm) - 1;
        const CollPath lq = {coll_shfl(q.sx, l), coll_shfl(q.sy, l), coll_shfl(q.sz, l), coll_shfl(q.rx, l),
                             coll_shfl(q.ry, l), coll_shfl(q.rz, l), coll_shfl(q.L, l)};
        const CollWords lw = {__shfl_sync(FULLW, w.a, l), __shfl_sync(FULLW, w.b, l), __shfl_sync(FULLW, w.c, l)};
        const CollBox lb = {__shfl_sync(FULLW, bx.lox, l), __shfl_sync(FULLW, bx.loy, l), __shfl_sync(FULLW, bx.loz, l),
                            __shfl_sync(FULLW, bx.hix, l), __shfl_sync(FULLW, bx.hiy, l), __shfl_sync(FULLW, bx.hiz, l)};
        Hits t = s.from(l);
        const unsigned tested = coll_wide(src.params(__shfl_sync(FULLW, cloth, l)), lq, lw, lb, t);
        if (gbase == l) s = t;
        if (COUNT_WIDE && lane == l) ntest += tested;
    }
}

// The response of every group's path S -> E (valid: whether it has one; o: its
// node's plane offset), G lanes per path; DEEP: see coll_cells.  True in the group's first lane if
// the node hits, with its position x; REC also records the response data.
template <bool REC, int G, bool DEEP, class Src>
__device__ __forceinline__ bool collide_path(const Src &src, int cloth, const StepParams &p, bool valid, float sx,
                                             float sy, float sz, float ex, float ey, float ez, long long o, float3 &x,
                                             unsigned &ntest)
{
    CollPath q = {};
    CollBox bx = {0, 0, 0, 0, 0, 0};
    CollWords w = {0u, 0u, 0u};
    int ncell = 0;
    bool wide = false;
    int2 run = make_int2(0, 0);
    if (valid) {
        bx = coll_box(p, sx, sy, sz, ex, ey, ez);
        if (DEEP) run = coll_run(p, bx.lox, bx.loy, bx.loz);  // loads while the direction is computed
        if (coll_path(p, sx, sy, sz, ex, ey, ez, q)) {
            w = coll_words(p, sx, sy, sz, ex, ey, ez, q);
            const long long nc = (long long)(bx.hix - bx.lox + 1) * (bx.hiy - bx.loy + 1) * (bx.hiz - bx.loz + 1);
            wide = nc > COLL_MAXC;
            ncell = wide ? 0 : (int)nc;
        }
    }
    NodeHits<REC> s = {};
    coll_cells<G, false, DEEP>(src, cloth, p, q, bx, w, run, ncell, wide, s, ntest);
    if (s.K == 0 || (threadIdx.x & 31) % G != 0) return false;
    const float m = s.acc / (float)s.K;
    // product and sum rounded separately, the same bits in every kernel
    x = make_float3(__fadd_rn(q.sx, __fmul_rn(m, q.rx)), __fadd_rn(q.sy, __fmul_rn(m, q.ry)),
                    __fadd_rn(q.sz, __fmul_rn(m, q.rz)));
    if constexpr (REC) coll_record(p, o, m, (float)s.K, q.rx, q.ry, q.rz, s.g1, s.g2);
    return true;
}

// A lane's first list entry and its path, loaded ahead by the kernel (p.parity
// is the substep's).  Any offset is taken: one outside the planes reads node 0.
struct CollFirst {
    int o;
    float sx, sy, sz, ex, ey, ez;

    __device__ __forceinline__ void load(const StepParams &p, int entry)
    {
        const long long st = p.stride;
        const float *in = (p.parity & 1) ? p.state1 : p.state0, *out = (p.parity & 1) ? p.state0 : p.state1;
        o = entry >= 0 && entry < st ? entry : 0;
        sx = __ldg(in + o); sy = __ldg(in + st + o); sz = __ldg(in + 2 * st + o);
        ex = out[o]; ey = out[st + o]; ez = out[2 * st + o];
    }
};

// One round of the list pass, G lanes per node: every group brings one entry
// (valid: whether it has one; i: its index for src.entry).  Src supplies
// entry(i, cloth, offset), params(cloth) and DEEP (see coll_cells).  ahead: the
// entry was loaded ahead (first; cloth 0).  ntest and nhit accumulate, in the
// group's first lane, the candidate triangles and whether the node hit.  REC:
// also records the hits' response data (coll_record).
template <bool REC, int G, class Src>
__device__ __forceinline__ void collide_round(const Src &src, unsigned long long k, bool valid, unsigned long long i,
                                              float &fsum, unsigned &ntest, unsigned &nhit, bool ahead,
                                              const CollFirst *first)
{
    int cloth = 0;
    long long o = 0;
    if (valid) {
        if (ahead) o = first->o;
        else src.entry(i, cloth, o);
    }
    const StepParams &p = src.params(cloth);
    const long long st = p.stride;
    const float *in = (k & 1ull) ? p.state1 : p.state0;
    float *out = (k & 1ull) ? p.state0 : p.state1;
    float sx = 0.0f, sy = 0.0f, sz = 0.0f, ex = 0.0f, ey = 0.0f, ez = 0.0f;
    if (ahead) {
        sx = first->sx; sy = first->sy; sz = first->sz;
        ex = first->ex; ey = first->ey; ez = first->ez;
    } else if (valid) {
        sx = __ldg(in + o); sy = __ldg(in + st + o); sz = __ldg(in + 2 * st + o);
        ex = out[o]; ey = out[st + o]; ez = out[2 * st + o];
    }
    float3 x;
    if (collide_path<REC, G, Src::DEEP>(src, cloth, p, valid, sx, sy, sz, ex, ey, ez, o, x, ntest)) {
        out[o] = x.x;
        out[st + o] = x.y;
        out[2 * st + o] = x.z;
        out[3 * st + o] *= p.restitution;
        out[4 * st + o] *= p.restitution;
        out[5 * st + o] *= p.restitution;
        fsum += x.x + x.y + x.z;
        nhit++;
    }
}

// The pass over a list of n entries in chunks of 32 / G neighbours, one per
// warp and round.  A list of fewer chunks than warps is dealt over the CTAs
// first (every SM gets some); a longer one in runs of COLL_WARPS chunks per
// CTA, so that a CTA's warps share the lines of the cells they read.
// ahead: the lane's entry of the first round with G = COLL_GMAX and fewer
// chunks than warps (index coll_first_index()), or null.
constexpr int COLL_GMAX = 8;
__device__ __forceinline__ unsigned coll_first_index()
{
    const unsigned c = (threadIdx.x >> 5) * gridDim.x + blockIdx.x;
    return c * (32 / COLL_GMAX) + (threadIdx.x & 31) / COLL_GMAX;
}
template <bool REC, int G, class Src>
__device__ __forceinline__ void collide_chunks(const Src &src, unsigned long long k, unsigned n, float &fsum,
                                               unsigned &ntest, unsigned &nhit, const CollFirst *ahead)
{
    constexpr unsigned PER = 32 / G;
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const unsigned chunks = (n + PER - 1u) / PER, nw = gridDim.x * COLL_WARPS;
    const bool deal = chunks < nw;
    const unsigned first = deal ? (unsigned)wib * gridDim.x + blockIdx.x : blockIdx.x * COLL_WARPS + wib;
    for (unsigned c = first; c < chunks; c += nw) {
        const unsigned long long i = (unsigned long long)PER * c + (unsigned)(lane / G);
        collide_round<REC, G>(src, k, i < n, i, fsum, ntest, nhit, G == COLL_GMAX && ahead && deal && c == first, ahead);
    }
}
// Lanes per node: a short list leaves most of the grid's lanes idle and is
// bound by its chain of dependent loads, so COLL_GMAX lanes share a node's
// candidates; two where that still takes one round; else one, which does
// the least work per node.  SHORT: the cloth is small (coll_short), so only
// the first form is compiled in.
template <bool REC, bool SHORT, class Src>
__device__ __forceinline__ void collide_list(const Src &src, unsigned long long k, unsigned n, float &fsum,
                                             unsigned &ntest, unsigned &nhit, const CollFirst *ahead = nullptr)
{
    const unsigned lanes = gridDim.x * 32u * COLL_WARPS;
    if (SHORT || n <= lanes / COLL_GMAX)
        collide_chunks<REC, COLL_GMAX>(src, k, n, fsum, ntest, nhit, ahead);
    else if (n <= lanes / 2u)
        collide_chunks<REC, 2>(src, k, n, fsum, ntest, nhit, nullptr);
    else
        collide_chunks<REC, 1>(src, k, n, fsum, ntest, nhit, nullptr);
}

// One thread of a CTA adds its counts to the cloth's running statistics.  The
// adds return nothing, so no thread waits on them.
__device__ __forceinline__ void coll_stats_store(DevCtrl *ctrl, unsigned listed, unsigned tested, unsigned hits)
{
    unsigned long long *q = ctrl->stat[blockIdx.x % CLOTH_STAT_SLOTS];
    if (listed) atomicAdd(q, (unsigned long long)listed);
    if (tested) atomicAdd(q + 1, (unsigned long long)tested);
    if (hits) atomicAdd(q + 2, (unsigned long long)hits);
}

// Adds a collision pass's counts to the cloth's running statistics: every
// warp's tested candidates and hit nodes are summed per CTA in shared memory
// (s2, zeroed by the caller before a __syncthreads), then one thread adds the
// CTA's totals; CTA 0 also adds the list length n.
__device__ __forceinline__ void coll_stats_add(DevCtrl *ctrl, unsigned *s2, unsigned n, unsigned ntest, unsigned nhit)
{
    const unsigned h = __reduce_add_sync(0xffffffffu, nhit), q = __reduce_add_sync(0xffffffffu, ntest);
    if ((threadIdx.x & 31) == 0) {
        atomicAdd(&s2[0], q);
        atomicAdd(&s2[1], h);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        coll_stats_store(ctrl, blockIdx.x == 0 ? n : 0u, s2[0], s2[1]);
    }
}

// ------------------------------------------- edge-triangle narrow phase
// The paper's own narrow phase (Section 3): edges of the cloth triangles (the
// grid's quads split along their (r,c)-(r+1,c+1) diagonal) at the updated
// positions against the surface triangles.  A hit of an edge at P affects
// every vertex of the cloth triangles that share the edge; an affected free
// node i gets the direction from its previous position S_i towards P,
// stopping delta short, max(|P - S_i| - delta, 0) (P - S_i)/|P - S_i|, and
// moves by the mean over its hits (Algorithm 2).  Gathered per node: the 12
// edges whose triangles contain node (r, c), each as (owner endpoint ->
// other endpoint) with the owner the edge's upper-left node, the orientation
// the test's arithmetic is defined in.
struct EdgeOfs {
    signed char ar, ac, br, bc;
};
__device__ __forceinline__ EdgeOfs edge_of_node(int q)
{
    // (0,+1) edges: own, left, up-left row above, row below
    // (+1,0) edges: own, above, up-left column, right column
    // (+1,+1) edges: own, up-left, the two that have (r,c) as opposite vertex
    switch (q) {
    case 0: return {0, 0, 0, 1};
    case 1: return {0, -1, 0, 0};
    case 2: return {-1, -1, -1, 0};
    case 3: return {1, 0, 1, 1};
    case 4: return {0, 0, 1, 0};
    case 5: return {-1, 0, 0, 0};
    case 6: return {-1, -1, 0, -1};
    case 7: return {0, 1, 1, 1};
    case 8: return {0, 0, 1, 1};
    case 9: return {-1, -1, 0, 0};
    case 10: return {-1, 0, 0, 1};
    default: return {0, -1, 1, 0};
    }
}
constexpr int EDGES_PER_NODE = 12;
// Hits after an edge's first whose points pass A stores (p.edge_more); pass B
// walks an edge with more hits than 1 + EDGE_MORE again.
constexpr int EDGE_MORE = CLOTH_EDGE_MORE;

// The kind of the triangulation edge from (ra, ca) to (rb, cb): 0 (0,+1),
// 1 (+1,0), 2 (+1,+1).
__device__ __forceinline__ int edge_kind(int ra, int ca, int rb, int cb) { return rb == ra ? 0 : (cb == ca ? 1 : 2); }

// An edge's hits (see NodeHits): rec = (the first hit's point, the number of
// hits); the points of hits 2 .. 1 + EDGE_MORE go to p.edge_more at the edge's slot.
struct EdgeHits {
    float4 rec;
    long long slot;

    __device__ __forceinline__ void one(const StepParams &p, const CollPath &q, float th)
    {
        const float3 P = coll_hit_point(q, th);
        if (rec.w == 0.0f) rec = make_float4(P.x, P.y, P.z, 0.0f);
        else if (rec.w <= (float)EDGE_MORE)
            p.edge_more[(long long)(rec.w - 1.0f) * 3 * p.stride + slot] = make_float4(P.x, P.y, P.z, 1.0f);
        rec.w += 1.0f;
    }
    template <int G>
    __device__ __forceinline__ void add(const StepParams &p, const CollPath &q, bool hit, float th, float, float,
                                        const float4 &, const float4 &)
    {
        if constexpr (G == 1) {
            if (hit) one(p, q, th);
        } else {
            const int lane = threadIdx.x & 31, gbase = lane & ~(G - 1);
            unsigned hm = (__ballot_sync(0xffffffffu, hit) >> gbase) & (0xffffffffu >> (32 - G));
            while (__any_sync(0xffffffffu, hm != 0u)) {
                const float ht = coll_shfl(th, hm ? gbase + __ffs((int)hm) - 1 : lane);
                if (hm) one(p, q, ht);  // every lane of the group stores the same point
                hm &= hm - 1u;
            }
        }
    }
    __device__ __forceinline__ EdgeHits from(int l) const
    {
        return {make_float4(coll_shfl(rec.x, l), coll_shfl(rec.y, l), coll_shfl(rec.z, l), coll_shfl(rec.w, l)),
                __shfl_sync(0xffffffffu, slot, l)};
    }
};

// Pass A of the edge narrow phase: every listed node tests the three edges it
// owns, (0,+1), (+1,0) and (+1,+1) from it (the triangulation's edges,
// oriented from their upper-left endpoint), at the updated positions, so each
// edge is tested once.  G lanes per edge as in the node pass; a warp's edges
// are of one kind.  Records per edge its first hit
// point (in candidate order) and its number of hits, p.edge_hit[kind * stride +
// owner] = (P, K), and the points of its hits 2 .. 1 + EDGE_MORE at
// p.edge_more[(h - 2) * 3 * stride + kind * stride + owner].  Counts the
// tested candidates and the edges that hit into ntest and nhit.  Against one
// that searched shared memory for each candidate: 256 x 256 nodes lying on
// 81,920 triangles 669 -> 329 us per step of cloth_step with its copies, falling
// onto them (steps 150 to 250) 276 -> 271.  Where edges are long the time is
// that of the slowest warp: a warp's edges from one place of the list made it
// 309 and 367, from 32 places 346 and 258; up to 18 cells per lane 338 (falling).
constexpr int EDGE_MAXC = 8;  // cells of an edge's box one lane goes through
template <int G>
__device__ __forceinline__ void edge_test_chunks(const StepParams &p, unsigned long long k, unsigned n,
                                                 unsigned &ntest, unsigned &nhit)
{
    constexpr unsigned PER = 32 / G;
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const long long st = p.stride;
    const float *xs = (k & 1ull) ? p.state0 : p.state1;  // updated positions (written by the walk)
    const unsigned per_kind = (n + PER - 1u) / PER, nw = gridDim.x * COLL_WARPS;
    const unsigned chunks = 3u * per_kind;  // three chunks of 32 edges per 32 nodes: far below 2^32
    const unsigned first = chunks < nw ? (unsigned)wib * gridDim.x + blockIdx.x : blockIdx.x * COLL_WARPS + wib;
    unsigned *next = p.ctrl->edge_next + (k & 1ull);
    // every warp has a first chunk; the others go to whoever is free, since edges
    // differ in their cells and hits (256 x 256 nodes are 1.3 chunks a warp: with
    // c += nw the pass took two full rounds, 90 against 80 us per substep; lists
    // of nodes keep c += nw, whose neighbours share an SM's L1: 4 % faster there)
    for (unsigned c = first; c < chunks;) {
        const int kind = (int)(c / per_kind);
        // long edges come in clusters, so a warp takes pairs of neighbours from
        // sixteen places of the list (a cluster in one warp held it for 100 us)
        const unsigned cc0 = c % per_kind;
        const unsigned i = G > 1 ? PER * cc0 + (unsigned)(lane / G)
                                 : (unsigned)(lane / 2) * 2u * per_kind + 2u * cc0 + (unsigned)(lane % 2);
        bool has = false, wide = false;
        int ncell = 0;
        CollPath path = {};
        CollBox bx = {0, 0, 0, 0, 0, 0};
        CollWords w = {0u, 0u, 0u};
        EdgeHits s = {make_float4(0.0f, 0.0f, 0.0f, 0.0f), 0};
        if (i < n) {
            const int o = __ldg(p.coll_list + i);
            const int r = o / p.pitch, cc = o - r * p.pitch;
            const int rb = r + (kind >= 1 ? 1 : 0), cb = cc + (kind != 1 ? 1 : 0);
            if (rb < p.ny && cb < p.nx) {
                has = true;
                s.slot = (long long)kind * st + o;
                const long long ob = (long long)rb * p.pitch + cb;
                const float x0 = xs[o], y0 = xs[st + o], z0 = xs[2 * st + o];
                const float x1 = xs[ob], y1 = xs[st + ob], z1 = xs[2 * st + ob];
                if (coll_path(p, x0, y0, z0, x1, y1, z1, path)) {
                    bx = coll_box(p, x0, y0, z0, x1, y1, z1);
                    w = coll_words(p, x0, y0, z0, x1, y1, z1, path);
                    const long long nc = (long long)(bx.hix - bx.lox + 1) * (bx.hiy - bx.loy + 1) * (bx.hiz - bx.loz + 1);
                    wide = nc > EDGE_MAXC;
                    ncell = wide ? 0 : (int)nc;
                }
            }
        }
        coll_cells<G, true, false>(OneCloth{p}, 0, p, path, bx, w, make_int2(0, 0), ncell, wide, s, ntest);
        if (has && lane % G == 0) {
            p.edge_hit[s.slot] = s.rec;
            nhit += s.rec.w > 0.0f ? 1u : 0u;
        }
        if (chunks <= nw) break;
        c = 0u;
        if (lane == 0) c = nw + atomicAdd(next, 1u);
        c = __shfl_sync(0xffffffffu, c, 0);
    }
}
__device__ __forceinline__ void edge_test_list(const StepParams &p, unsigned long long k, unsigned n, unsigned &ntest,
                                               unsigned &nhit)
{
    const unsigned lanes = gridDim.x * 32u * COLL_WARPS;
    if (3u * n <= lanes / COLL_GMAX) edge_test_chunks<COLL_GMAX>(p, k, n, ntest, nhit);
    else edge_test_chunks<1>(p, k, n, ntest, nhit);
}

// Running sum of one node's response directions (Algorithm 2): adds the
// direction from S towards the hit point P, stopping delta short.
struct EdgeAcc {
    float ax, ay, az;
    int K;
};
__device__ __forceinline__ void edge_acc_add(EdgeAcc &a, float delta, float sx, float sy, float sz, float Px,
                                             float Py, float Pz)
{
    const float wx = Px - sx, wy = Py - sy, wz = Pz - sz;
    const float lw = sqrtf(wx * wx + wy * wy + wz * wz);
    const float sc = lw > 0.0f ? fmaxf(lw - delta, 0.0f) / lw : 0.0f;
    a.ax += sc * wx;
    a.ay += sc * wy;
    a.az += sc * wz;
    a.K++;
}

// An edge with more hits than pass A stored: walks its candidates again, in
// order and behind the same filter (the hits must be pass A's, also where
// rounding alone decides), and adds every hit after the first (already added).
// Out of line: rare, and it keeps the gather's unrolled loop small.
static __device__ __noinline__ EdgeAcc edge_rewalk(const StepParams &p, const float *xs, long long oa, long long ob,
                                                   float sx, float sy, float sz, EdgeAcc a)
{
    const long long st = p.stride;
    const float x0 = xs[oa], y0 = xs[st + oa], z0 = xs[2 * st + oa];
    const float x1 = xs[ob], y1 = xs[st + ob], z1 = xs[2 * st + ob];
    CollPath path;
    if (!coll_path(p, x0, y0, z0, x1, y1, z1, path)) return a;
    const CollBox bx = coll_box(p, x0, y0, z0, x1, y1, z1);
    const CollWords w = coll_words(p, x0, y0, z0, x1, y1, z1, path);
    bool first = true;
    for (int cz = bx.loz; cz <= bx.hiz; cz++)
        for (int cy = bx.loy; cy <= bx.hiy; cy++)
            for (int cx = bx.lox; cx <= bx.hix; cx++) {
                const long long cell = ((long long)cz * p.gd[1] + cy) * p.gd[0] + cx;
                const int e0 = __ldg(p.cell_start + cell), e1 = __ldg(p.cell_start + cell + 1);
                const unsigned need = coll_need(bx, cx, cy, cz);
                for (int ee = e0; ee < e1; ee++) {
                    float th, over, f;
                    float4 A, B, C;
                    if (!coll_overlap(__ldg(p.efil + ee), w, need)) continue;
                    if (!coll_candidate(p, path, ee, cx, cy, cz, bx.lox, bx.loy, bx.loz, th, over, f, A, B, C)) continue;
                    if (first) {
                        first = false;
                        continue;
                    }
                    const float3 hp = coll_hit_point(path, th);
                    edge_acc_add(a, p.delta, sx, sy, sz, hp.x, hp.y, hp.z);
                }
            }
    return a;
}

// Pass B: every listed free node gathers the hits of the 12 edges whose
// triangles contain it (in the order of edge_of_node, each edge's hits in
// candidate order) and writes its response to p.edge_resp[i]: (position, 1),
// or zeros without a hit.  An edge whose owner was not listed this substep
// (stamp) cannot hit.  The stamps, then the records, of the 12 edges are
// loaded before any is used; an edge with more than 1 + EDGE_MORE hits is
// walked again (edge_rewalk).
__device__ __forceinline__ void edge_gather_list(const StepParams &p, unsigned long long k, unsigned n)
{
    const long long st = p.stride;
    const float *in = (k & 1ull) ? p.state1 : p.state0;
    const float *xs = (k & 1ull) ? p.state0 : p.state1;
    const unsigned long long stamp = k + 1ull;
    for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const int o = __ldg(p.coll_list + i);
        const bool pinned = p.pin_bits && ((__ldg(p.pin_bits + (o >> 5)) >> (o & 31)) & 1u);
        float4 resp = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        if (!pinned) {
            const int r = o / p.pitch, c = o - r * p.pitch;
            const float sx = __ldg(in + o), sy = __ldg(in + st + o), sz = __ldg(in + 2 * st + o);
            bool live[EDGES_PER_NODE];
#pragma unroll
            for (int q = 0; q < EDGES_PER_NODE; q++) {
                const EdgeOfs e = edge_of_node(q);
                const int ra = r + e.ar, ca = c + e.ac, rb = r + e.br, cb = c + e.bc;
                const bool inside = ra >= 0 && ca >= 0 && rb < p.ny && cb < p.nx && ca < p.nx && cb >= 0;
                live[q] = inside && p.edge_stamp[inside ? (long long)ra * p.pitch + ca : 0] == stamp;
            }
            float4 rec[EDGES_PER_NODE];
#pragma unroll
            for (int q = 0; q < EDGES_PER_NODE; q++) {
                const EdgeOfs e = edge_of_node(q);
                const long long slot = (long long)edge_kind(e.ar, e.ac, e.br, e.bc) * st +
                                       (long long)(r + e.ar) * p.pitch + (c + e.ac);
                rec[q] = live[q] ? p.edge_hit[slot] : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            }
            EdgeAcc acc = {0.0f, 0.0f, 0.0f, 0};
#pragma unroll
            for (int q = 0; q < EDGES_PER_NODE; q++) {
                const float4 rq = rec[q];
                if (rq.w == 0.0f) continue;
                edge_acc_add(acc, p.delta, sx, sy, sz, rq.x, rq.y, rq.z);
                if (rq.w == 1.0f) continue;
                const EdgeOfs e = edge_of_node(q);
                const long long oa = (long long)(r + e.ar) * p.pitch + (c + e.ac);
                if (rq.w <= (float)(1 + EDGE_MORE)) {
                    const long long slot = (long long)edge_kind(e.ar, e.ac, e.br, e.bc) * st + oa;
                    for (int h = 1; h < (int)rq.w; h++) {
                        const float4 P = p.edge_more[(long long)(h - 1) * 3 * st + slot];
                        edge_acc_add(acc, p.delta, sx, sy, sz, P.x, P.y, P.z);
                    }
                } else {
                    const long long ob = (long long)(r + e.br) * p.pitch + (c + e.bc);
                    acc = edge_rewalk(p, xs, oa, ob, sx, sy, sz, acc);
                }
            }
            if (acc.K > 0)
                resp = make_float4(sx + acc.ax / (float)acc.K, sy + acc.ay / (float)acc.K, sz + acc.az / (float)acc.K,
                                   1.0f);
        }
        p.edge_resp[i] = resp;
    }
}
