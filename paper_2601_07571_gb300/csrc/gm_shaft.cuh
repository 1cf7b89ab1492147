// gm_shaft.cuh -- occlusion of the rays of one warp as one shaft, and the warp-tile body built on it.
//
// All rays that a warp traces for one fixation leave one eye toward 32 neighbouring samples, so they
// fill a thin pyramid (the shaft). The warp walks the 4-wide tree once for the shaft, all lanes on
// boxes: per step up to 8 nodes of a shared-memory stack are popped and each lane tests one child box
// of one of them against the interval of ray directions; surviving inner children are pushed, those
// that the shaft enters later below the nearer ones, and leaves are collected. Once SH_FLUSH triangles
// are collected (or the stack is empty) the lanes turn to rays: each lane loads one triangle relative
// to the eye and its box in the image plane, every ray marks the triangles whose image box holds it,
// and tests those with the watertight test of the per-ray walk (same arithmetic on the same
// differences). Occluded rays leave the shaft, which shrinks; the walk ends with the last of them.
//
// Why: a warp of per-ray walks issued about 6900 instructions per (tile, fixation) at the
// 800k-triangle scene with 16 of 32 lanes active -- the lanes' walks end at different times and meet
// their leaves at different steps. The same 34 nodes and 4 triangles per ray, shared by 30 rays, are
// 16 steps and about 90 collected triangles of a shaft, of which a ray tests 3.3 after the image-box
// test.
#pragma once

#include <type_traits>

#include "gm_trace.cuh"

namespace {

// Collected triangles that are tested at once: few the first time (most shafts end on the first surface
// they meet), more after that.
constexpr int SH_FLUSH = 16, SH_FLUSH2 = 24;
constexpr int SH_CAND = 56;     // below SH_FLUSH2 before a step, and a step collects up to 32
// Triangles tested against one shaft before its rays walk the binary tree one by one: where triangles
// are much smaller than the spacing of the samples, a shaft holds thousands that no ray meets.
constexpr int SH_BUDGET = 640;
// Stack entries. Above SH_WIDE one node is popped per step, so from there the stack grows by at most 3
// per level of the tree, which has at most 33 levels (the build refuses a binary tree deeper than 64):
// SH_WIDE - 8 + 32 + 99 <= SH_STACK, and no step needs a check.
constexpr int SH_WIDE = 128;
constexpr int SH_STACK = 256;

struct ShaftWarp {
    float4 tri[32 * 3];         // collected triangles: vertices relative to the eye, axes permuted; A.w = triangle id
    float4 box[32];             // their image boxes (x0, x1, y0, y1)
    int stack[SH_STACK];
    uint32_t cand[SH_CAND];     // leaf slots
};

__device__ __forceinline__ float rcp_approx(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// The interval of ray directions as slab coefficients. With l and h a box's bounds relative to the eye
// on one axis and d in [lo, hi], t d can reach [l, h] only for t >= l P and t >= h M (the bound that
// does not apply is <= 0, or huge where no direction goes that way), and only for t <= x Q + C with
// x = h, or l where all directions are negative (C huge where the interval holds 0).
struct Shaft {
    float P[3], M[3], Q[3], C[3];
    bool neg[3];
};

// From each lane's bounds of its rays' directions (an empty lane: +inf, -inf).
__device__ __forceinline__ void set_shaft(Shaft& S, const float lo_l[3], const float hi_l[3]) {
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const float lo = redux_min(lo_l[k]), hi = redux_max(hi_l[k]);
        const float il = rcp_approx(lo), ih = rcp_approx(hi);
        S.P[k] = hi > 0.f ? ih : 1e30f;
        S.M[k] = lo < 0.f ? il : -1e30f;
        S.neg[k] = hi < 0.f;
        S.Q[k] = lo > 0.f ? il : (hi < 0.f ? ih : 0.f);
        S.C[k] = lo > 0.f || hi < 0.f ? 0.f : 1e30f;
    }
}

__device__ __forceinline__ void set_shaft(Shaft& S, bool in, float dx, float dy, float dz) {
    const float lo[3] = {in ? dx : INFINITY, in ? dy : INFINITY, in ? dz : INFINITY};
    const float hi[3] = {in ? dx : -INFINITY, in ? dy : -INFINITY, in ? dz : -INFINITY};
    set_shaft(S, lo, hi);
}

// The per-ray walk of a shaft that is over its budget (out of line: rare, and its registers are its own).
__device__ __noinline__ bool shaft_ray_hit(float ex, float ey, float ez, float dx, float dy, float dz, float tmax,
                                           uint32_t own, const float4* __restrict__ nodes,
                                           const float4* __restrict__ tris, uint32_t nt, int* __restrict__ err,
                                           uint32_t* __restrict__ n_tri) {
    Ray R;
    make_ray(R, make_float3(ex, ey, ez), make_float3(dx, dy, dz), tmax);
    int hit = -1;
    uint32_t nn = 0;
    return occluded(R, own, nodes, tris, nt, err, nn, *n_tri, hit);
}

// The watertight test of a ray whose dominant axis is not the shaft's: in its own axes, from vertices kept
// in the axes (rx, ry, the third).
__device__ __forceinline__ bool other_axes_hit(const float3 d, int rx, int ry, float4 A, float4 B, float4 C, float tmax) {
    const float ax = fabsf(d.x), ay = fabsf(d.y), az = fabsf(d.z);
    const int kz = (ax > ay) ? (ax > az ? 0 : 2) : (ay > az ? 1 : 2);
    const int k1 = kz == 2 ? 0 : kz + 1, k2 = k1 == 2 ? 0 : k1 + 1;
    const float dk = comp(d, kz);
    const int kx = dk < 0.f ? k2 : k1, ky = dk < 0.f ? k1 : k2;
    auto at = [&](const float4& v, int k) { return k == rx ? v.x : (k == ry ? v.y : v.z); };
    return tri_core(at(A, kx), at(A, ky), at(A, kz), at(B, kx), at(B, ky), at(B, kz), at(C, kx), at(C, ky), at(C, kz),
                    comp(d, kx) / dk, comp(d, ky) / dk, 1.0f / dk, tmax);
}

// What the walks of all shafts that end at one tile start from: the tree opened along the nodes that
// overlap the tile's box, as up to 32 subtrees and leaves (lo, link), (hi, -). One step over it takes the
// place of the first steps from the root, which have few boxes to test.
struct ShaftStart {
    float4 box[32][2];
    int n;
};

// One warp builds the list for the box [lo, hi] of its tile. Nodes to open wait with their boxes in
// `open` (32 entries of 2 float4); a step opens as many (at most 8) as the list can hold the children of.
__device__ __forceinline__ void shaft_start(const float lo[3], const float hi[3], const float4* __restrict__ nodes4,
                                            const float4* __restrict__ tris, const uint32_t nt, float4* open,
                                            ShaftStart& F) {
    const int lane = threadIdx.x & 31;
    const unsigned lt = gm_lanemask_lt();
    const int j = lane >> 2;
    int n = 0, m = 0;   // listed, waiting
    bool root = nt > 1;
    if (!root) {        // one triangle: a leaf whose box every shaft enters
        if (lane == 0) {
            F.box[0][0] = make_float4(-INFINITY, -INFINITY, -INFINITY, __int_as_float(~0));
            F.box[0][1] = make_float4(INFINITY, INFINITY, INFINITY, 0.f);
        }
        n = 1;
    }
    while (root || m > 0) {
        const int take = root ? 1 : min(min(m, 8), (32 - n - m) / 3);   // each opened node may add 3 entries
        if (take == 0) break;
        const bool act = j < take;
        const int node = !act || root ? 0 : __float_as_int(open[2 * (m - 1 - j)].w);
        if (!root) m -= take;
        root = false;
        const float4* N = nodes4 + 8 * (size_t)node + 2 * (lane & 3);
        const float4 a = __ldg(N), b = __ldg(N + 1);
        const int link = __float_as_int(a.w);
        const bool have = act && link != LINK_EMPTY;
        const bool in = have && link >= 0 && a.x <= hi[0] && b.x >= lo[0] && a.y <= hi[1] && b.y >= lo[1] &&
                        a.z <= hi[2] && b.z >= lo[2];
        const unsigned hm = __ballot_sync(0xffffffffu, have), im = __ballot_sync(0xffffffffu, in);
        __syncwarp();
        const int bi = __popc(im & lt), bo = __popc(hm & ~im & lt);
        if (in) {
            open[2 * (m + bi)] = a;
            open[2 * (m + bi) + 1] = b;
        } else if (have) {
            F.box[n + bo][0] = a;
            F.box[n + bo][1] = b;
        }
        m += __popc(im);
        n += __popc(hm & ~im);
        __syncwarp();
    }
    if (lane < m) {   // still to open: listed as they are
        F.box[n + lane][0] = open[2 * lane];
        F.box[n + lane][1] = open[2 * lane + 1];
    }
    if (lane == 0) F.n = n + m;
}

// One box per lane against the shaft from the eye e; entered leaves are collected (nc of them), entered
// inner nodes pushed (sp).
__device__ __forceinline__ void shaft_step(const Shaft& S, const float ex, const float ey, const float ez,
                                       const float tbox, const bool act, const float4 a, const float4 b, ShaftWarp& W,
                                       int& sp, int& nc) {
    const int lane = threadIdx.x & 31;
    const unsigned lt = gm_lanemask_lt();
    const int link = __float_as_int(a.w);
    const float lx = a.x - ex, ly = a.y - ey, lz = a.z - ez;
    const float hx = b.x - ex, hy = b.y - ey, hz = b.z - ez;
    const float en = fmax3(fmax3(lx * S.P[0], hx * S.M[0], ly * S.P[1]),
                           fmax3(hy * S.M[1], lz * S.P[2], hz * S.M[2]), 0.f);
    const float out = fmin3(fmaf(S.neg[0] ? lx : hx, S.Q[0], S.C[0]), fmaf(S.neg[1] ? ly : hy, S.Q[1], S.C[1]),
                            fminf(fmaf(S.neg[2] ? lz : hz, S.Q[2], S.C[2]), tbox));
    // 1e-5 covers the rounding of the differences and coefficients (the boxes' own margin covers the
    // per-ray test's)
    const bool hit = act && en * 0.99999f <= out && link != LINK_EMPTY;
    const bool inner = hit && link >= 0;
    const unsigned hm = __ballot_sync(0xffffffffu, hit), im = __ballot_sync(0xffffffffu, inner);
    const int before_i = __popc(im & lt);
    if (hit && link < 0) W.cand[nc + __popc(hm & lt) - before_i] = (uint32_t)~link;
    nc += __popc(hm & ~im);
    if (im) {
        // children entered later than the others (by the mean of the bit patterns, which order
        // like the non-negative entries) go below them
        const int cnt = __popc(im);
        const int q = inner ? __float_as_int(en) >> 5 : 0;
        const int sum = __reduce_add_sync(0xffffffffu, q);
        const unsigned fm = __ballot_sync(0xffffffffu, inner && q * cnt > sum);
        const int before_f = __popc(fm & lt);
        if (inner) W.stack[sp + ((fm >> lane) & 1u ? before_f : __popc(fm) + before_i - before_f)] = link;
        sp += cnt;
    }
    __syncwarp();
}

// The m triangles of W.cand from entry `at` on, one per lane: vertices relative to the eye in the axes
// (rx, ry, rz), and their image boxes on the side sgn of rz.
__device__ __forceinline__ void shaft_collect(const float ex, const float ey, const float ez, const int rx, const int ry,
                                              const int rz, const float sgn, const float4* __restrict__ tris, const int at,
                                              const int m, ShaftWarp& W) {
    const int lane = threadIdx.x & 31;
    float4 bb = make_float4(INFINITY, -INFINITY, INFINITY, -INFINITY);
    if (lane < m) {
        const uint32_t slot = W.cand[at + lane];
        const float4 a = __ldg(&tris[3 * (size_t)slot]), b = __ldg(&tris[3 * (size_t)slot + 1]);
        const float4 c = __ldg(&tris[3 * (size_t)slot + 2]);
        const float3 A = make_float3(a.x - ex, a.y - ey, a.z - ez);
        const float3 B = make_float3(b.x - ex, b.y - ey, b.z - ez);
        const float3 Cc = make_float3(c.x - ex, c.y - ey, c.z - ez);
        const float4 pa = make_float4(comp(A, rx), comp(A, ry), comp(A, rz), a.w);
        const float4 pb = make_float4(comp(B, rx), comp(B, ry), comp(B, rz), 0.f);
        const float4 pc = make_float4(comp(Cc, rx), comp(Cc, ry), comp(Cc, rz), 0.f);
        W.tri[3 * lane] = pa;
        W.tri[3 * lane + 1] = pb;
        W.tri[3 * lane + 2] = pc;
        const float zmin = fmin3(pa.z * sgn, pb.z * sgn, pc.z * sgn);
        const float side = fmax3(fmaxf(fabsf(pa.x), fabsf(pa.y)), fmaxf(fabsf(pb.x), fabsf(pb.y)),
                                 fmaxf(fabsf(pc.x), fabsf(pc.y)));
        if (zmin * 1e6f > side) {
            const float ia = rcp_approx(pa.z), ib = rcp_approx(pb.z), ic = rcp_approx(pc.z);
            const float x0 = fmin3(pa.x * ia, pb.x * ib, pc.x * ic), x1 = fmax3(pa.x * ia, pb.x * ib, pc.x * ic);
            const float y0 = fmin3(pa.y * ia, pb.y * ib, pc.y * ic), y1 = fmax3(pa.y * ia, pb.y * ib, pc.y * ic);
            // 2^-18 (1 + |X| + |Y|)^2 bounds the rounding of the image points and of the
            // watertight test (the eye grid's margin)
            const float r = 1.f + fmaxf(fabsf(x0), fabsf(x1)) + fmaxf(fabsf(y0), fabsf(y1));
            const float mg = r * r * (1.f / 262144.f);
            bb = make_float4(x0 - mg, x1 + mg, y0 - mg, y1 + mg);
        } else {   // reaches the plane through the eye: no bounded image
            bb = make_float4(-INFINITY, INFINITY, -INFINITY, INFINITY);
        }
    }
    W.box[lane] = bb;
    __syncwarp();
}

// Whether the segment e -> e + d of every lane with `in` set is unoccluded (false for the others). All
// lanes of the warp call it, at least one with `in`. (dx, dy, dz) = sample - eye. n_node counts for the
// warp (the same in every lane), n_tri per lane.
__device__ __forceinline__ bool shaft_visible(bool in, const float dx, const float dy, const float dz,
                                              const uint32_t own, const float ex, const float ey, const float ez,
                                              const ShaftStart& F, const float4* __restrict__ nodes,
                                              const float4* __restrict__ nodes4, const float4* __restrict__ tris,
                                              const uint32_t nt, const float tmax, ShaftWarp& W, int* __restrict__ err,
                                              uint32_t& n_node, uint32_t& n_tri) {
    const int lane = threadIdx.x & 31;
    const unsigned lt = gm_lanemask_lt();
    const float3 d = make_float3(dx, dy, dz);
    // the watertight test's axes of this lane's ray, and of the first ray: triangles are kept in those
    const float ax = fabsf(dx), ay = fabsf(dy), az = fabsf(dz);
    const int kz = (ax > ay) ? (ax > az ? 0 : 2) : (ay > az ? 1 : 2);
    const bool back = comp(d, kz) < 0.f;
    unsigned alive = __ballot_sync(0xffffffffu, in);
    const int src = __ffs(alive) - 1;
    const int rz = __shfl_sync(0xffffffffu, kz, src);
    const bool rback = __shfl_sync(0xffffffffu, (int)back, src) != 0;
    const int r1 = rz == 2 ? 0 : rz + 1, r2 = r1 == 2 ? 0 : r1 + 1;
    const int rx = rback ? r2 : r1, ry = rback ? r1 : r2;
    const bool uni = __all_sync(0xffffffffu, !in || (kz == rz && back == rback));
    const float dz_r = comp(d, rz);
    const float qx = comp(d, rx) / dz_r, qy = comp(d, ry) / dz_r, qz = 1.0f / dz_r;
    const float sgn = rback ? -1.f : 1.f;
    Shaft S;
    set_shaft(S, in, dx, dy, dz);
    const float tbox = tmax * 1.0001f;
    int sp = 0, nc = 0, budget = SH_BUDGET, flush = SH_FLUSH;
    shaft_step(S, ex, ey, ez, tbox, lane < F.n, F.box[lane][0], F.box[lane][1], W, sp, nc);
    for (;;) {
        while (nc < flush && sp > 0) {
            const int take = sp > SH_WIDE ? 1 : min(sp, 8);
            const bool act = (lane >> 2) < take;
            const int node = act ? W.stack[sp - 1 - (lane >> 2)] : 0;
            sp -= take;
            n_node += (uint32_t)take;
            const float4* N = nodes4 + 8 * (size_t)node + 2 * (lane & 3);
            shaft_step(S, ex, ey, ez, tbox, act, __ldg(N), __ldg(N + 1), W, sp, nc);
        }
        flush = SH_FLUSH2;
        const unsigned before = alive;
        while (nc > 0) {
            const int m = min(nc, 32);
            nc -= m;
            budget -= m;
            shaft_collect(ex, ey, ez, rx, ry, rz, sgn, tris, nc, m, W);
            unsigned mask = 0;
            for (int c0 = 0; c0 < m; c0 += 8) {
                unsigned mk = 0;
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    const float4 t = W.box[c0 + c];
                    if (qx >= t.x && qx <= t.y && qy >= t.z && qy <= t.w) mk |= 1u << c;
                }
                mask |= mk << c0;
            }
            // a ray without an image point on the first ray's side is tested against every triangle
            if (!uni && !(dz_r * sgn > 0.f)) mask = m == 32 ? 0xffffffffu : (1u << m) - 1u;
            if (!in) mask = 0;
            if (uni) {
                while (mask) {
                    const int c = __ffs(mask) - 1;
                    mask &= mask - 1u;
                    ++n_tri;
                    const float4 A = W.tri[3 * c];
                    if (__float_as_uint(A.w) == own) continue;
                    const float4 B = W.tri[3 * c + 1], Cc = W.tri[3 * c + 2];
                    if (tri_core(A.x, A.y, A.z, B.x, B.y, B.z, Cc.x, Cc.y, Cc.z, qx, qy, qz, tmax)) {
                        in = false;
                        mask = 0;
                    }
                }
            } else {
                // the rays' dominant axes differ: each in its own axes, from the permuted vertices
                const int k1 = kz == 2 ? 0 : kz + 1, k2 = k1 == 2 ? 0 : k1 + 1;
                const int kx = back ? k2 : k1, ky = back ? k1 : k2;
                const float dk = comp(d, kz);
                const float sx = comp(d, kx) / dk, sy = comp(d, ky) / dk, sz = 1.0f / dk;
                auto at = [&](const float4& v, int k) { return k == rx ? v.x : (k == ry ? v.y : v.z); };
                while (mask) {
                    const int c = __ffs(mask) - 1;
                    mask &= mask - 1u;
                    ++n_tri;
                    const float4 A = W.tri[3 * c];
                    if (__float_as_uint(A.w) == own) continue;
                    const float4 B = W.tri[3 * c + 1], Cc = W.tri[3 * c + 2];
                    if (tri_core(at(A, kx), at(A, ky), at(A, kz), at(B, kx), at(B, ky), at(B, kz), at(Cc, kx), at(Cc, ky),
                                 at(Cc, kz), sx, sy, sz, tmax)) {
                        in = false;
                        mask = 0;
                    }
                }
            }
            alive = __ballot_sync(0xffffffffu, in);
            if (alive == 0) return false;
            __syncwarp();
        }
        if (sp == 0) return in;
        if (budget <= 0) {
            uint32_t tested = 0;
            if (in) in = !shaft_ray_hit(ex, ey, ez, dx, dy, dz, tmax, own, nodes, tris, nt, err, &tested);
            n_tri += tested;
            __syncwarp();
            return in;
        }
        if (alive != before) set_shaft(S, in, dx, dy, dz);
    }
}

// The same for a tile of 32 NS samples, NS rays per lane: bit k of `in` asks for the segment to sample
// 32 k + lane of `pos` (positions, own triangle in w), the same bit of the result says that it is
// unoccluded. All lanes of the warp call it, at least one with a bit set.
template <int NS>
__device__ __forceinline__ unsigned shaft_visible_wide(unsigned in, const float4* pos, const float ex, const float ey,
                                                  const float ez, const ShaftStart& F, const float4* __restrict__ nodes,
                                                  const float4* __restrict__ nodes4, const float4* __restrict__ tris,
                                                  const uint32_t nt, const float tmax, ShaftWarp& W,
                                                  int* __restrict__ err, uint32_t& n_node, uint32_t& n_tri) {
    const int lane = threadIdx.x & 31;
    auto dir = [&](int k) {   // sample - eye
        const float4 p = pos[32 * k + lane];
        return make_float3(p.x - ex, p.y - ey, p.z - ez);
    };
    // the watertight test's axis and side of a ray: 2 x axis + (side < 0)
    auto axis_of = [&](const float3 d) {
        const float ax = fabsf(d.x), ay = fabsf(d.y), az = fabsf(d.z);
        const int kz = (ax > ay) ? (ax > az ? 0 : 2) : (ay > az ? 1 : 2);
        return 2 * kz + (comp(d, kz) < 0.f ? 1 : 0);
    };
    // triangles are kept in the axes of the first ray; rays share them unless a tile straddles a diagonal
    const unsigned lanes_in = __ballot_sync(0xffffffffu, in != 0u);
    const int mine = axis_of(dir(in ? __ffs(in) - 1 : 0));
    const int ref = __shfl_sync(0xffffffffu, mine, __ffs(lanes_in) - 1);
    const int rz = ref >> 1;
    const int r1 = rz == 2 ? 0 : rz + 1, r2 = r1 == 2 ? 0 : r1 + 1;
    const int rx = ref & 1 ? r2 : r1, ry = ref & 1 ? r1 : r2;
    const float sgn = ref & 1 ? -1.f : 1.f;
    float qx[NS], qy[NS], qz[NS];
    uint32_t own[NS];
    Shaft S;
    bool same = true;
    auto bound = [&](float lo[3], float hi[3]) {   // of the directions of this lane's rays
#pragma unroll
        for (int c = 0; c < 3; ++c) lo[c] = INFINITY, hi[c] = -INFINITY;
#pragma unroll
        for (int k = 0; k < NS; ++k) {
            if (!((in >> k) & 1u)) continue;
            const float3 d = dir(k);
            lo[0] = fminf(lo[0], d.x), lo[1] = fminf(lo[1], d.y), lo[2] = fminf(lo[2], d.z);
            hi[0] = fmaxf(hi[0], d.x), hi[1] = fmaxf(hi[1], d.y), hi[2] = fmaxf(hi[2], d.z);
        }
    };
#pragma unroll
    for (int k = 0; k < NS; ++k) {
        const float3 d = dir(k);
        const float dz = comp(d, rz);
        qx[k] = comp(d, rx) / dz;
        qy[k] = comp(d, ry) / dz;
        qz[k] = dz == 0.f ? 0.f : 1.0f / dz;   // 0: no image point (never a ray in its own axes)
        own[k] = __float_as_uint(pos[32 * k + lane].w);
        same = same && (!((in >> k) & 1u) || axis_of(d) == ref);
    }
    const bool uni = __all_sync(0xffffffffu, same);
    {
        float lo[3], hi[3];
        bound(lo, hi);
        set_shaft(S, lo, hi);
    }
    const float tbox = tmax * 1.0001f;
    int sp = 0, nc = 0, budget = SH_BUDGET, flush = SH_FLUSH;
    shaft_step(S, ex, ey, ez, tbox, lane < F.n, F.box[lane][0], F.box[lane][1], W, sp, nc);
    for (;;) {
        while (nc < flush && sp > 0) {
            const int take = sp > SH_WIDE ? 1 : min(sp, 8);
            const bool act = (lane >> 2) < take;
            const int node = act ? W.stack[sp - 1 - (lane >> 2)] : 0;
            sp -= take;
            n_node += (uint32_t)take;
            const float4* N = nodes4 + 8 * (size_t)node + 2 * (lane & 3);
            shaft_step(S, ex, ey, ez, tbox, act, __ldg(N), __ldg(N + 1), W, sp, nc);
        }
        flush = SH_FLUSH2;
        const unsigned before = in;
        while (nc > 0) {
            const int m = min(nc, 32);
            nc -= m;
            budget -= m;
            shaft_collect(ex, ey, ez, rx, ry, rz, sgn, tris, nc, m, W);
            // the triangles whose image box holds each ray
            unsigned mask[NS];
#pragma unroll
            for (int k = 0; k < NS; ++k) mask[k] = 0;
            for (int c0 = 0; c0 < m; c0 += 8) {
                unsigned mk[NS];
#pragma unroll
                for (int k = 0; k < NS; ++k) mk[k] = 0;
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    const float4 t = W.box[c0 + c];
#pragma unroll
                    for (int k = 0; k < NS; ++k)
                        if (qx[k] >= t.x && qx[k] <= t.y && qy[k] >= t.z && qy[k] <= t.w) mk[k] |= 1u << c;
                }
#pragma unroll
                for (int k = 0; k < NS; ++k) mask[k] |= mk[k] << c0;
            }
            unsigned any = 0;
#pragma unroll
            for (int k = 0; k < NS; ++k) {
                // a ray without an image point on the first ray's side is tested against every triangle
                if (!uni && !(qz[k] * sgn > 0.f)) mask[k] = m == 32 ? 0xffffffffu : (1u << m) - 1u;
                if (!((in >> k) & 1u)) mask[k] = 0;
                any |= mask[k];
            }
            // each lane takes its rays' triangles one after another
            auto test = [&](auto one_axis) {
                while (any) {
                    int r = 0;
                    unsigned mk = mask[0];
                    float x = qx[0], y = qy[0], z = qz[0];
                    uint32_t o = own[0];
#pragma unroll
                    for (int k = 1; k < NS; ++k) {
                        const bool next = mk == 0u;
                        r = next ? k : r;
                        mk = next ? mask[k] : mk;
                        x = next ? qx[k] : x;
                        y = next ? qy[k] : y;
                        z = next ? qz[k] : z;
                        o = next ? own[k] : o;
                    }
                    const int c = __ffs(mk) - 1;
                    mk &= mk - 1u;
                    ++n_tri;
                    const float4 A = W.tri[3 * c];
                    if (__float_as_uint(A.w) != o) {
                        const float4 Bv = W.tri[3 * c + 1], Cv = W.tri[3 * c + 2];
                        bool hit;
                        if constexpr (decltype(one_axis)::value)
                            hit = tri_core(A.x, A.y, A.z, Bv.x, Bv.y, Bv.z, Cv.x, Cv.y, Cv.z, x, y, z, tmax);
                        else
                            hit = other_axes_hit(dir(r), rx, ry, A, Bv, Cv, tmax);
                        if (hit) {
                            in &= ~(1u << r);
                            mk = 0;
                        }
                    }
                    any = mk;
                    mask[0] = r == 0 ? mk : mask[0];
#pragma unroll
                    for (int k = 1; k < NS; ++k) {
                        mask[k] = r == k ? mk : mask[k];
                        any |= mask[k];
                    }
                }
            };
            if (uni) test(std::true_type{});
            else test(std::false_type{});
            if (!__any_sync(0xffffffffu, in != 0u)) return 0u;
            __syncwarp();
        }
        if (sp == 0) return in;
        if (budget <= 0) {
            uint32_t tested = 0;
            for (int k = 0; k < NS; ++k) {
                if (!((in >> k) & 1u)) continue;
                const float3 d = dir(k);
                if (shaft_ray_hit(ex, ey, ez, d.x, d.y, d.z, tmax, __float_as_uint(pos[32 * k + lane].w), nodes, tris, nt,
                                  err, &tested))
                    in &= ~(1u << k);
            }
            n_tri += tested;
            __syncwarp();
            return in;
        }
        if (__any_sync(0xffffffffu, in != before)) {
            float lo[3], hi[3];
            bound(lo, hi);
            set_shaft(S, lo, hi);
        }
    }
}

// ---- blocks of warps on warp tiles -----------------------------------------------------------------
// A block takes a warp tile (32 consecutive work-order samples) through the whole fixation list, in
// batches: first the fixations whose cones reach the tile's bounding sphere are listed, in order; then
// the warps trace them, one (tile, fixation) at a time whichever warp is free, each leaving a 32-bit mask
// of visible samples; then one warp adds the visible weights, in list order, to the tile's compensated
// sums. All warps of the block share a tile that sees many rays (a gazed patch, a patch of tiny
// triangles), sample sets of a few thousand fill the GPU, and the sums stay those of a sequential pass.
// (A tile per warp with shared lists instead: 126 ms against 68 ms at the 800k-triangle scene, whose
// patch of 1 mm triangles then falls to few blocks.)
// Fixations are listed until a batch has shaft_fill of them (or none is left), shaft_per a thread at a
// step. Smaller batches wait for their last item more often: a wide tile's at 1 instead of 128 takes
// 33 ms at the city's windows instead of 21, a narrow tile's at 64 or 128 instead of 256 more as well.
constexpr int SH_FILL1 = 256, SH_FILL4 = 128;
__host__ __device__ constexpr int shaft_fill(int ns) { return ns == 1 ? SH_FILL1 : SH_FILL4; }
__host__ __device__ constexpr int shaft_per(int ns, int nt) { return ns == 1 && nt == ACC_THREADS ? 2 : 1; }
__host__ __device__ constexpr int shaft_list(int ns, int nt) { return shaft_fill(ns) - 1 + shaft_per(ns, nt) * nt; }

template <int NS, int NT = ACC_THREADS>
struct ShaftBlock {
    ShaftWarp warp[NT / 32];
    ShaftStart start;
    float4 pos[NS == 1 ? 1 : 32 * NS];   // the tile's samples (NS = 1: in registers)
    uint32_t list[shaft_list(NS, NT)];      // fixation indices
    uint32_t vis[NS][shaft_list(NS, NT)];   // visible samples of each item
    uint32_t pass[NT / 32];    // passing fixations of each warp's 32 shaft_per in one fill step
    int next;                   // next item to trace
};

// The cone test and weight of sample p for fixation (F0, F1); in-cone and weight.
__device__ __forceinline__ bool cone_test(const float4 p, const float4 F0, const float4 F1, const float K, float& px,
                                          float& py, float& pz, float& c2, float& d1s) {
    px = p.x - F0.x, py = p.y - F0.y, pz = p.z - F0.z;
    const float d1 = fmaf(px, F1.x, fmaf(py, F1.y, pz * F1.z));
    const float cx = fmaf(py, F1.z, -pz * F1.y);
    const float cy = fmaf(pz, F1.x, -px * F1.z);
    const float cz = fmaf(px, F1.y, -py * F1.x);
    c2 = fmaf(cx, cx, fmaf(cy, cy, cz * cz));
    d1s = d1 * d1;
    return d1 > 0.f && c2 <= K * d1s;
}

// The weight is rounded on its own (never fused into the compensated sum): every form adds the same value.
__device__ __forceinline__ float cone_weight(const float w, const float c2, const float d1s, const float C2) {
    return __fmul_rn(w, ex2_approx(-C2 * __fdividef(c2, d1s)));
}

__device__ __forceinline__ float4 work_sample(const float4* __restrict__ spos, uint32_t j, uint32_t ns) {
    // padding lanes hold NaN positions: every cone test on them is false
    return j < ns ? spos[j] : make_float4(__int_as_float(0x7fc00000), 0.f, 0.f, __uint_as_float(0xffffffffu));
}

// The box of the warp's samples from each lane's bounds, and the sphere around it.
__device__ __forceinline__ float4 tile_sphere(float lo[3], float hi[3]) {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        lo[c] = redux_min(lo[c]);
        hi[c] = redux_max(hi[c]);
    }
    return make_float4(0.5f * (lo[0] + hi[0]), 0.5f * (lo[1] + hi[1]), 0.5f * (lo[2] + hi[2]),
                       0.5f * sqrtf((hi[0] - lo[0]) * (hi[0] - lo[0]) + (hi[1] - lo[1]) * (hi[1] - lo[1]) +
                                    (hi[2] - lo[2]) * (hi[2] - lo[2])) * 1.0001f);
}

// The 128 threads of half h of a block wait for one another (barrier 0 is the block's).
__device__ __forceinline__ void half_sync(int h) { asm volatile("bar.sync %0, 128;" ::"r"(h + 1) : "memory"); }

// One block, all threads: tile `tile` (32 NS consecutive work-order samples) against fixations [0, nf) of
// `fix` (packed (e, w), (r^, window), sorted by window). A window's sums are written when the next visible
// fixation opens another one, or at the end.
// HALF: by the 128 threads of one half of a block (0 or 1), on its own barrier.
template <bool DEBUG, int NS, int NT = ACC_THREADS, bool HALF = false>
__device__ __forceinline__ void shaft_tile(const uint32_t tile, const float4* __restrict__ spos,
                                           const uint32_t* __restrict__ sidx, const float4* __restrict__ fix,
                                           const uint32_t nf, const float4* __restrict__ nodes,
                                           const float4* __restrict__ nodes4, const float4* __restrict__ tris,
                                           const AccParams& P, float* __restrict__ out,
                                           unsigned int* __restrict__ max_bits, ShaftBlock<NS, NT>& B,
                                           unsigned long long* __restrict__ dbg_cursor, const DebugOut& dbg,
                                           int* __restrict__ err, TileStats& st) {
    const int tid = HALF ? threadIdx.x & (NT - 1) : threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const unsigned lt = gm_lanemask_lt();
    auto sync = [&]() {
        if constexpr (HALF) half_sync(threadIdx.x / NT);
        else __syncthreads();
    };
    const uint32_t j0 = tile * (32u * NS) + lane;
    float lo[3] = {INFINITY, INFINITY, INFINITY}, hi[3] = {-INFINITY, -INFINITY, -INFINITY};
    uint32_t n_live = 0;   // of this lane
    float4 p0;             // NS = 1: the lane's sample
#pragma unroll
    for (int k = 0; k < NS; ++k) {
        const float4 p = work_sample(spos, j0 + 32 * k, P.ns);
        if (NS == 1) p0 = p;
        else if (warp == 0) B.pos[32 * k + lane] = p;
        if (j0 + 32 * k < P.ns) {
            ++n_live;
            lo[0] = fminf(lo[0], p.x), lo[1] = fminf(lo[1], p.y), lo[2] = fminf(lo[2], p.z);
            hi[0] = fmaxf(hi[0], p.x), hi[1] = fmaxf(hi[1], p.y), hi[2] = fmaxf(hi[2], p.z);
        }
    }
    float4 bs = tile_sphere(lo, hi);
    if (warp == 0) shaft_start(lo, hi, nodes4, tris, P.nt, B.warp[0].tri, B.start);
    if (!P.tile_cull) bs.w = -1.f;
    // warp k < NS keeps the sums of samples 32 k + lane
    const uint32_t j = j0 + 32 * warp;
    const bool live = warp < NS && j < P.ns;
    float sum = 0.f, cmp = 0.f;
    uint32_t cur = 0xffffffffu;
    uint32_t n_in = 0, n_vis = 0, n_node = 0, n_tri = 0, n_items = 0;
    auto flush = [&](uint32_t w) {
        if (live && (P.W == 1 || sum != 0.f)) out[(size_t)w * P.ns + sidx[j]] = sum;
        const float m = redux_max(sum);
        if (lane == 0 && m > 0.f) atomicMax(&max_bits[w], __float_as_uint(m));
        sum = 0.f;
        cmp = 0.f;
    };
    for (uint32_t pos = 0; pos < nf;) {
        // list the fixations that reach the tile: a warp takes 32 PER consecutive ones of each step
        constexpr int PER = shaft_per(NS, NT);
        int cnt = 0;
        while (cnt < shaft_fill(NS) && pos < nf) {
            unsigned reach[PER];
            int mine = 0;
#pragma unroll
            for (int r = 0; r < PER; ++r) {
                const uint32_t i = pos + (warp * PER + r) * 32 + lane;
                reach[r] = __ballot_sync(0xffffffffu, i < nf && cone_reaches_sphere(bs, __ldg(&fix[2 * i]),
                                                                                    __ldg(&fix[2 * i + 1]), P.tanphi));
                mine += __popc(reach[r]);
            }
            if (lane == 0) B.pass[warp] = mine;
            sync();
            const int n = lane < NT / 32 ? (int)B.pass[lane] : 0;
            int at = cnt + __reduce_add_sync(0xffffffffu, lane < warp ? n : 0);
            cnt += __reduce_add_sync(0xffffffffu, n);
#pragma unroll
            for (int r = 0; r < PER; ++r) {
                if ((reach[r] >> lane) & 1u) B.list[at + __popc(reach[r] & lt)] = pos + (warp * PER + r) * 32 + lane;
                at += __popc(reach[r]);
            }
            pos += PER * NT;
            if (tid == 0) B.next = 0;
            sync();
        }
        if (warp == 0) n_items += cnt;
        // trace the items
        for (;;) {
            int k = 0;
            if (lane == 0) k = atomicAdd(&B.next, 1);
            k = __shfl_sync(0xffffffffu, k, 0);
            if (k >= cnt) break;
            const uint32_t i = B.list[k];
            const float4 F0 = __ldg(&fix[2 * i]), F1 = __ldg(&fix[2 * i + 1]);
            float px, py, pz, c2, d1s;
            unsigned in = 0, vis = 0;
            if constexpr (NS == 1) {
                const bool one = cone_test(p0, F0, F1, P.K, px, py, pz, c2, d1s);
                if (__any_sync(0xffffffffu, one)) {
                    in = one;
                    vis = shaft_visible(one, px, py, pz, __float_as_uint(p0.w), F0.x, F0.y, F0.z, B.start, nodes, nodes4,
                                        tris, P.nt, P.tmax, B.warp[warp], err, n_node, n_tri);
                }
            } else {
#pragma unroll
                for (int r = 0; r < NS; ++r)
                    in |= cone_test(B.pos[32 * r + lane], F0, F1, P.K, px, py, pz, c2, d1s) ? 1u << r : 0u;
                if (__any_sync(0xffffffffu, in != 0u))
                    vis = shaft_visible_wide<NS>(in, B.pos, F0.x, F0.y, F0.z, B.start, nodes, nodes4, tris, P.nt, P.tmax,
                                                 B.warp[warp], err, n_node, n_tri);
            }
            n_in += __popc(in);
            n_vis += __popc(vis);
            if (DEBUG) {
                for (int r = 0; r < NS; ++r) {
                    if (!((in >> r) & 1u)) continue;
                    cone_test(NS == 1 ? p0 : B.pos[32 * r + lane], F0, F1, P.K, px, py, pz, c2, d1s);
                    record_pair(dbg_cursor, dbg, P, sidx, tile * (32u * NS), 32u, 32 * r + lane, i, (vis >> r) & 1u,
                                cone_weight(F0.w, c2, d1s, P.C2));
                }
            }
#pragma unroll
            for (int r = 0; r < NS; ++r) {
                const unsigned vm = __ballot_sync(0xffffffffu, (vis >> r) & 1u);
                if (lane == 0) B.vis[r][k] = vm;
            }
        }
        sync();
        // add the visible weights in list order
        if (warp < NS) {
            const float4 p = NS == 1 ? p0 : B.pos[32 * warp + lane];
            for (int k0 = 0; k0 < cnt; k0 += 32) {
                const uint32_t mv = k0 + lane < cnt ? B.vis[warp][k0 + lane] : 0u;
                const uint32_t mi = k0 + lane < cnt ? B.list[k0 + lane] : 0u;
                unsigned todo = __ballot_sync(0xffffffffu, mv != 0u);
                while (todo) {
                    const int k = __ffs(todo) - 1;
                    todo &= todo - 1u;
                    const uint32_t i = __shfl_sync(0xffffffffu, mi, k), vm = __shfl_sync(0xffffffffu, mv, k);
                    const float4 F0 = __ldg(&fix[2 * i]), F1 = __ldg(&fix[2 * i + 1]);
                    const uint32_t win = __float_as_uint(F1.w);
                    if (win != cur) {
                        if (cur != 0xffffffffu) flush(cur);
                        cur = win;
                    }
                    if ((vm >> lane) & 1u) {
                        float px, py, pz, c2, d1s;
                        cone_test(p, F0, F1, P.K, px, py, pz, c2, d1s);
                        const float g = cone_weight(F0.w, c2, d1s, P.C2);
                        const float y = g - cmp;
                        const float t = sum + y;
                        cmp = (t - sum) - y;
                        sum = t;
                    }
                    __syncwarp();
                }
            }
        }
        sync();
    }
    if (warp < NS) {
        if (cur != 0xffffffffu) flush(cur);
        else if (P.W == 1) flush(0);   // nothing visible: window 0 is written as zeros
    }
    st.n_in += n_in;
    st.n_vis += n_vis;
    st.n_node += lane == 0 ? n_node : 0u;
    st.n_tri += n_tri;
    st.n_tested += (unsigned long long)n_live * n_items;
}

}  // namespace
