// gm_scene.cu -- gm_build_scene: meshes -> world triangles -> BVH; gm_scene_pose: re-posed meshes.
//
// The paper tests occlusion with a z-buffer rendered per point of view (Section 3.2.2); here
// occlusion is an exact segment test against every triangle, accelerated by a binary BVH built
// on the GPU in data-parallel steps:
//   1. world vertices: FP64 transform per vertex, rounded to FP32 (same operation order as
//      the FP64 reference: ((m0 x + m1 y) + m2 z) + m3, no fused multiply-add);
//   2. 63-bit Morton code of each triangle centroid in the centroid bounds;
//   3. stable radix sort of the codes (leaf order);
//   4. the hierarchy, by one of two builders:
//      PLOC (default; Meister & Bittner, "Parallel locally-ordered clustering for bounding volume
//      hierarchy construction", TVCG 2018): rounds of nearest-neighbour search by union-box
//      surface area within +-8 positions of the Morton order, merging of mutual pairs and
//      compaction, until one cluster is left;
//      LBVH (Karras, "Maximizing parallelism in the construction of BVHs, octrees, and k-d
//      trees", HPG 2012): one thread per internal node finds its key range and split, then a
//      bottom-up refit in which the second child to arrive writes the node's union box;
//   5. internal nodes renumbered in depth-first order (a parent's nearer child is often in the
//      next 64 bytes).
// Node layout (64 B): the boxes of both children plus the two child links, so one node fetch
// decides both children. A child link >= 0 is an internal node, < 0 is leaf ~link (one
// triangle). Boxes are widened by 2^-19 of the scene's largest coordinate so that the FP32
// slab test never rejects a triangle the watertight triangle test would hit.
// Dynamic scenes keep the mesh-local triangles; gm_scene_pose recomputes the world triangles for
// new transforms and refits every box bottom-up over the unchanged hierarchy.
#include <cmath>
#include <cstring>
#include <string>
#include <vector>

#include "gm_internal.cuh"
#include "gm_scan.cuh"

namespace {

// Clustering radius of the PLOC builder: 8 neighbours on each side traced the paper scene in
// 244 ms against 257 ms for 16 (34.2 vs 34.1 nodes per ray; the depth-first layout of the
// smaller-radius tree caches better), and builds faster.
constexpr int kPlocRadius = 8;

struct Mat16 {
    double m[16];
};

__global__ void k_transform(const float* __restrict__ v, uint32_t nv, Mat16 M, float* __restrict__ out) {
    uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nv) return;
    double x = v[3 * i], y = v[3 * i + 1], z = v[3 * i + 2];
#pragma unroll
    for (int r = 0; r < 3; ++r) {
        double s = __dadd_rn(__dmul_rn(M.m[4 * r + 0], x), __dmul_rn(M.m[4 * r + 1], y));
        s = __dadd_rn(s, __dmul_rn(M.m[4 * r + 2], z));
        s = __dadd_rn(s, M.m[4 * r + 3]);
        out[3 * i + r] = __double2float_rn(s);
    }
}

__device__ __forceinline__ unsigned int f2ord(float f) {
    unsigned int b = __float_as_uint(f);
    return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}
__device__ __forceinline__ float ord2f(unsigned int o) {
    return __uint_as_float((o & 0x80000000u) ? (o & 0x7fffffffu) : ~o);
}

// bounds layout (ordered-uint encoded floats): [0..2] centroid min, [3..5] centroid max,
// [6..8] vertex min, [9..11] vertex max.
__global__ void k_bounds_init(unsigned int* b) {
    int i = threadIdx.x;
    if (i < 12) b[i] = ((i / 3) % 2 == 0) ? 0xffffffffu : 0u;
}

// Fold the block's centroid (0..2) and vertex (3..5) boxes into the scene's: one atomic per block and
// bound (one per warp and bound, all on the same 12 words, took 150 of k_gather's 197 us at 800k
// triangles). All 256 threads call it.
__device__ __forceinline__ void fold_bounds(const float lo[6], const float hi[6], unsigned int* __restrict__ bounds) {
    __shared__ unsigned int slo[6], shi[6];
    if (threadIdx.x < 6) {
        slo[threadIdx.x] = 0xffffffffu;
        shi[threadIdx.x] = 0u;
    }
    __syncthreads();
#pragma unroll
    for (int c = 0; c < 6; ++c) {
        const unsigned int l = f2ord(redux_min(lo[c])), h = f2ord(redux_max(hi[c]));
        if ((threadIdx.x & 31) == 0) {
            atomicMin(&slo[c], l);
            atomicMax(&shi[c], h);
        }
    }
    __syncthreads();
    if (threadIdx.x < 6) {
        const int at = threadIdx.x < 3 ? threadIdx.x : threadIdx.x + 3;
        atomicMin(&bounds[at], slo[threadIdx.x]);
        atomicMax(&bounds[at + 3], shi[threadIdx.x]);
    }
}

__global__ void k_gather(const float* __restrict__ wv, const uint32_t* __restrict__ idx, uint32_t nt,
                         uint32_t nv, uint32_t tri_base, uint32_t mesh, float4* __restrict__ tri_canon,
                         uint32_t* __restrict__ tri_mesh, unsigned int* __restrict__ bounds,
                         int* __restrict__ err) {
    uint32_t t = blockIdx.x * blockDim.x + threadIdx.x;
    float lo[6], hi[6];
#pragma unroll
    for (int c = 0; c < 6; ++c) { lo[c] = INFINITY; hi[c] = -INFINITY; }
    if (t < nt) {
        float3 v[3];
        bool bad = false;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            uint32_t vi = idx[3 * t + k];
            if (vi >= nv) { bad = true; vi = 0; }
            v[k] = make_float3(wv[3 * vi], wv[3 * vi + 1], wv[3 * vi + 2]);
        }
        if (bad) atomicCAS(err, 0, GM_DEV_BAD_INDEX);
        uint32_t g = tri_base + t;
        tri_canon[3 * g + 0] = make_float4(v[0].x, v[0].y, v[0].z, 0.f);
        tri_canon[3 * g + 1] = make_float4(v[1].x, v[1].y, v[1].z, 0.f);
        tri_canon[3 * g + 2] = make_float4(v[2].x, v[2].y, v[2].z, 0.f);
        tri_mesh[g] = mesh;
        float c[3] = {(v[0].x + v[1].x + v[2].x) * (1.f / 3.f), (v[0].y + v[1].y + v[2].y) * (1.f / 3.f),
                      (v[0].z + v[1].z + v[2].z) * (1.f / 3.f)};
        const float* vf = &v[0].x;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            lo[a] = hi[a] = c[a];
            lo[3 + a] = fminf(fminf(vf[a], vf[3 + a]), vf[6 + a]);
            hi[3 + a] = fmaxf(fmaxf(vf[a], vf[3 + a]), vf[6 + a]);
        }
    }
    fold_bounds(lo, hi, bounds);
}

__device__ __forceinline__ uint64_t spread3_21(uint32_t v) {
    uint64_t x = v & 0x1fffffu;
    x = (x | x << 32) & 0x1f00000000ffffull;
    x = (x | x << 16) & 0x1f0000ff0000ffull;
    x = (x | x << 8) & 0x100f00f00f00f00full;
    x = (x | x << 4) & 0x10c30c30c30c30c3ull;
    x = (x | x << 2) & 0x1249249249249249ull;
    return x;
}

__device__ __forceinline__ uint32_t quant21(float c, float lo, float hi) {
    float ext = hi - lo;
    if (!(ext > 0.f)) return 0u;
    float q = (c - lo) / ext * 2097152.f;
    q = fminf(fmaxf(q, 0.f), 2097151.f);
    return (uint32_t)q;
}

__global__ void k_morton(const float4* __restrict__ tri, uint32_t nt, const unsigned int* __restrict__ bounds,
                         uint64_t* __restrict__ keys, uint32_t* __restrict__ vals) {
    uint32_t t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= nt) return;
    float4 a = tri[3 * t], b = tri[3 * t + 1], c = tri[3 * t + 2];
    float cx = (a.x + b.x + c.x) * (1.f / 3.f), cy = (a.y + b.y + c.y) * (1.f / 3.f),
          cz = (a.z + b.z + c.z) * (1.f / 3.f);
    uint32_t qx = quant21(cx, ord2f(bounds[0]), ord2f(bounds[3]));
    uint32_t qy = quant21(cy, ord2f(bounds[1]), ord2f(bounds[4]));
    uint32_t qz = quant21(cz, ord2f(bounds[2]), ord2f(bounds[5]));
    keys[t] = (spread3_21(qx) << 2) | (spread3_21(qy) << 1) | spread3_21(qz);
    vals[t] = t;
}

__device__ __forceinline__ int lcp(const uint64_t* __restrict__ keys, int n, int i, int j) {
    if (j < 0 || j >= n) return -1;
    uint64_t a = keys[i], b = keys[j];
    if (a != b) return __clzll((long long)(a ^ b));
    return 64 + __clz(i ^ j);
}

__global__ void k_hierarchy(const uint64_t* __restrict__ keys, int n, float4* __restrict__ nodes,
                            int* __restrict__ parent_node, int* __restrict__ parent_leaf) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n - 1) return;
    int d = (lcp(keys, n, i, i + 1) - lcp(keys, n, i, i - 1)) >= 0 ? 1 : -1;
    int dmin = lcp(keys, n, i, i - d);
    int lmax = 2;
    while (lcp(keys, n, i, i + lmax * d) > dmin) lmax <<= 1;
    int l = 0;
    for (int t = lmax >> 1; t >= 1; t >>= 1)
        if (lcp(keys, n, i, i + (l + t) * d) > dmin) l += t;
    int j = i + l * d;
    int dnode = lcp(keys, n, i, j);
    int s = 0, t = l;
    do {
        t = (t + 1) >> 1;
        if (lcp(keys, n, i, i + (s + t) * d) > dnode) s += t;
    } while (t > 1);
    int split = i + s * d + min(d, 0);
    int lo = min(i, j), hi = max(i, j);
    int left = (lo == split) ? ~split : split;
    int right = (hi == split + 1) ? ~(split + 1) : split + 1;
    nodes[4 * i + 3] = make_float4(__int_as_float(left), __int_as_float(right), 0.f, 0.f);
    if (left < 0) parent_leaf[~left] = i; else parent_node[left] = i;
    if (right < 0) parent_leaf[~right] = i; else parent_node[right] = i;
    if (i == 0) parent_node[0] = -1;
}

__device__ __forceinline__ void store_child_box(float* node, int side, const float lo[3], const float hi[3]) {
    // side 0: floats 0..5 = Lmin xyz, Lmax xyz; side 1: floats 6..11 = Rmin xyz, Rmax xyz
    float* p = node + 6 * side;
    p[0] = lo[0]; p[1] = lo[1]; p[2] = lo[2];
    p[3] = hi[0]; p[4] = hi[1]; p[5] = hi[2];
}

__global__ void k_refit(const float4* __restrict__ tri_canon, const uint32_t* __restrict__ order, int n,
                        float4* __restrict__ nodes, const int* __restrict__ parent_node,
                        const int* __restrict__ parent_leaf, unsigned int* __restrict__ flags,
                        const unsigned int* __restrict__ bounds, float4* __restrict__ bvh_tris) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    uint32_t t = order[i];
    float4 a = tri_canon[3 * t], b = tri_canon[3 * t + 1], c = tri_canon[3 * t + 2];
    bvh_tris[3 * i + 0] = make_float4(a.x, a.y, a.z, __uint_as_float(t));
    bvh_tris[3 * i + 1] = b;
    bvh_tris[3 * i + 2] = c;
    if (n == 1) return;
    float big = 0.f;
#pragma unroll
    for (int k = 0; k < 3; ++k) big = fmaxf(big, fmaxf(fabsf(ord2f(bounds[6 + k])), fabsf(ord2f(bounds[9 + k]))));
    const float margin = big * (1.0f / 524288.0f) + 1e-30f;
    float lo[3] = {fminf(fminf(a.x, b.x), c.x) - margin, fminf(fminf(a.y, b.y), c.y) - margin,
                   fminf(fminf(a.z, b.z), c.z) - margin};
    float hi[3] = {fmaxf(fmaxf(a.x, b.x), c.x) + margin, fmaxf(fmaxf(a.y, b.y), c.y) + margin,
                   fmaxf(fmaxf(a.z, b.z), c.z) + margin};
    int p = parent_leaf[i];
    int self = ~i;
    while (p >= 0) {
        float* node = reinterpret_cast<float*>(nodes + 4 * p);
        int left = __float_as_int(node[12]);
        store_child_box(node, left == self ? 0 : 1, lo, hi);
        __threadfence();
        if (atomicAdd(&flags[p], 1u) == 0u) return;  // the sibling finishes this node
        __threadfence();
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            lo[k] = fminf(__ldcg(node + k), __ldcg(node + 6 + k));
            hi[k] = fmaxf(__ldcg(node + 3 + k), __ldcg(node + 9 + k));
        }
        self = p;
        p = parent_node[p];
    }
}

constexpr int LINK_EMPTY = (int)0x80000000;

__device__ __forceinline__ void child_box(const float* node, int side, float lo[3], float hi[3]) {
    const float* p = node + 6 * side;
    lo[0] = p[0]; lo[1] = p[1]; lo[2] = p[2];
    hi[0] = p[3]; hi[1] = p[4]; hi[2] = p[5];
}

__global__ void k_collapse4(const float4* __restrict__ nodes, int n_int, const int64_t* __restrict__ incl,
                            float4* __restrict__ nodes4) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n_int) return;
    const int64_t before = i > 0 ? incl[i - 1] : 0;
    if (incl[i] == before) return;                    // odd depth: absorbed by its parent
    const int j = (int)before;                        // index of this 4-wide node
    const float* bn = reinterpret_cast<const float*>(nodes + 4 * i);
    float lo[4][3], hi[4][3];
    int link[4];
    int m = 0;
    for (int side = 0; side < 2; ++side) {
        const int c = __float_as_int(bn[12 + side]);
        if (c < 0) {
            child_box(bn, side, lo[m], hi[m]);
            link[m++] = c;
        } else {
            const float* cn = reinterpret_cast<const float*>(nodes + 4 * c);
            for (int s2 = 0; s2 < 2; ++s2) {
                const int g = __float_as_int(cn[12 + s2]);
                child_box(cn, s2, lo[m], hi[m]);
                link[m++] = g < 0 ? g : (int)(g > 0 ? incl[g - 1] : 0);
            }
        }
    }
    for (; m < 4; ++m) {
        for (int k = 0; k < 3; ++k) lo[m][k] = hi[m][k] = 1e30f;   // a box no segment reaches
        link[m] = LINK_EMPTY;
    }
    float4* o = nodes4 + 8 * (size_t)j;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        o[2 * k] = make_float4(lo[k][0], lo[k][1], lo[k][2], __int_as_float(link[k]));
        o[2 * k + 1] = make_float4(hi[k][0], hi[k][1], hi[k][2], 0.f);
    }
}

// ---- PLOC: parallel locally-ordered clustering (Meister & Bittner, TVCG 2018) ----------------
// Clusters start as the Morton-ordered leaves. Each round, every cluster finds the cluster within
// +-R positions whose union box has the smallest surface area; mutual nearest neighbours merge
// into a new node (the lower position keeps the merged cluster), and the array is compacted.
// Node indices are handed out downwards from n - 2, in position order, so the last merge -- the root --
// is node 0. A cluster is two float4: (lo, id) and (hi, leaves below).
//
// A round is two kernels: k_ploc_pair (neighbours, with a halo so that a block decides its own pairs, and
// the number of clusters that leave each block) and k_ploc_apply (nodes and compaction; a block sums the
// counts of the blocks before it). The cluster count stays on the device: the host launches PLOC_BATCH
// rounds at a time with the grid of the last count it read, rounds that find PLOC_TAIL clusters or
// fewer do nothing, and one block runs all remaining rounds in shared memory. At 800k triangles 100
// rounds of six kernels and a host read each took 3.4 ms of a 4.9 ms build; these take 0.7 ms.
constexpr int PLOC_T = 256;
constexpr int PLOC_P = 512;        // positions per block
constexpr int PLOC_TAIL = 1024;
constexpr int PLOC_BATCH = 12;

__device__ __forceinline__ float union_area(const float4 al, const float4 ah, const float4 bl, const float4 bh) {
    const float dx = fmaxf(ah.x, bh.x) - fminf(al.x, bl.x);
    const float dy = fmaxf(ah.y, bh.y) - fminf(al.y, bl.y);
    const float dz = fmaxf(ah.z, bh.z) - fminf(al.z, bl.z);
    return dx * dy + dy * dz + dz * dx;
}

__global__ void k_ploc_init(const float4* __restrict__ tri_canon, const uint32_t* __restrict__ order, int n,
                            const unsigned int* __restrict__ bounds, float4* __restrict__ blo,
                            float4* __restrict__ bhi, float4* __restrict__ bvh_tris, int* __restrict__ m_of) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    if (i == 0) m_of[0] = n;
    uint32_t t = order[i];
    float4 a = tri_canon[3 * t], b = tri_canon[3 * t + 1], c = tri_canon[3 * t + 2];
    bvh_tris[3 * i + 0] = make_float4(a.x, a.y, a.z, __uint_as_float(t));
    bvh_tris[3 * i + 1] = b;
    bvh_tris[3 * i + 2] = c;
    float big = 0.f;
#pragma unroll
    for (int k = 0; k < 3; ++k) big = fmaxf(big, fmaxf(fabsf(ord2f(bounds[6 + k])), fabsf(ord2f(bounds[9 + k]))));
    const float margin = big * (1.0f / 524288.0f) + 1e-30f;
    blo[i] = make_float4(fminf(fminf(a.x, b.x), c.x) - margin, fminf(fminf(a.y, b.y), c.y) - margin,
                         fminf(fminf(a.z, b.z), c.z) - margin, __int_as_float(~i));
    bhi[i] = make_float4(fmaxf(fmaxf(a.x, b.x), c.x) + margin, fmaxf(fmaxf(a.y, b.y), c.y) + margin,
                         fmaxf(fmaxf(a.z, b.z), c.z) + margin, __int_as_float(1));
}

// Nearest neighbour of cluster i (shared-memory position p) among positions i - R .. i + R of [0, m); the
// lowest position wins a tie. -1: none.
template <int R>
__device__ __forceinline__ int ploc_nearest(const float4* sl, const float4* sh, int p, int i, int m) {
    const float4 al = sl[p], ah = sh[p];
    float best = INFINITY;
    int bj = -1;
#pragma unroll 4
    for (int d = -R; d <= R; ++d) {
        const int j = i + d;
        if (d == 0 || j < 0 || j >= m) continue;
        const float a = union_area(al, ah, sl[p + d], sh[p + d]);
        if (a < best) {
            best = a;
            bj = j;
        }
    }
    return bj;
}

// Node k from the clusters at positions i < j; returns the merged cluster in (al, ah).
__device__ __forceinline__ void ploc_node(int k, float4& al, float4& ah, const float4 bl, const float4 bh,
                                          float4* __restrict__ nodes, int* __restrict__ parent_node,
                                          int* __restrict__ parent_leaf, unsigned int* __restrict__ leaves) {
    const int ci = __float_as_int(al.w), cj = __float_as_int(bl.w);
    const int n = __float_as_int(ah.w) + __float_as_int(bh.w);
    nodes[4 * (size_t)k + 0] = make_float4(al.x, al.y, al.z, ah.x);
    nodes[4 * (size_t)k + 1] = make_float4(ah.y, ah.z, bl.x, bl.y);
    nodes[4 * (size_t)k + 2] = make_float4(bl.z, bh.x, bh.y, bh.z);
    nodes[4 * (size_t)k + 3] = make_float4(al.w, bl.w, 0.f, 0.f);
    if (ci < 0) parent_leaf[~ci] = k; else parent_node[ci] = k;
    if (cj < 0) parent_leaf[~cj] = k; else parent_node[cj] = k;
    leaves[k] = (unsigned int)n;
    al = make_float4(fminf(al.x, bl.x), fminf(al.y, bl.y), fminf(al.z, bl.z), __int_as_float(k));
    ah = make_float4(fmaxf(ah.x, bh.x), fmaxf(ah.y, bh.y), fmaxf(ah.z, bh.z), __int_as_float(n));
}

// pair[i]: the position that i merges with, or -1; gone[block]: clusters of the block that leave (the
// upper ones of their pairs).
template <int R>
__global__ void __launch_bounds__(PLOC_T) k_ploc_pair(const int* __restrict__ m_of, const float4* __restrict__ blo,
                                                      const float4* __restrict__ bhi, int* __restrict__ pair,
                                                      int* __restrict__ gone) {
    __shared__ float4 sl[PLOC_P + 4 * R], sh[PLOC_P + 4 * R];
    __shared__ int snn[PLOC_P + 2 * R];
    __shared__ int count;
    const int m = *m_of, b0 = blockIdx.x * PLOC_P;
    if (m <= PLOC_TAIL || b0 >= m) return;
    if (threadIdx.x == 0) count = 0;
    for (int k = threadIdx.x; k < PLOC_P + 4 * R; k += PLOC_T) {
        const int g = b0 - 2 * R + k;
        if (g >= 0 && g < m) {
            sl[k] = blo[g];
            sh[k] = bhi[g];
        }
    }
    __syncthreads();
    for (int q = threadIdx.x; q < PLOC_P + 2 * R; q += PLOC_T) {
        const int i = b0 - R + q;
        snn[q] = i >= 0 && i < m ? ploc_nearest<R>(sl, sh, q + R, i, m) : -1;
    }
    __syncthreads();
    for (int q = threadIdx.x; q < PLOC_P; q += PLOC_T) {   // whole warps
        const int i = b0 + q;
        int p = -1;
        if (i < m) {
            const int j = snn[q + R];
            if (j >= 0 && snn[j - b0 + R] == i) p = j;
            pair[i] = p;
        }
        const unsigned up = __ballot_sync(0xffffffffu, p >= 0 && p < i);
        if ((threadIdx.x & 31) == 0 && up) atomicAdd(&count, __popc(up));
    }
    __syncthreads();
    if (threadIdx.x == 0) gone[blockIdx.x] = count;
}

__global__ void __launch_bounds__(PLOC_T) k_ploc_apply(const int* __restrict__ m_of, int* __restrict__ m_next,
                                                       const float4* __restrict__ blo, const float4* __restrict__ bhi,
                                                       const int* __restrict__ pair, const int* __restrict__ gone,
                                                       float4* __restrict__ blo2, float4* __restrict__ bhi2,
                                                       float4* __restrict__ nodes, int* __restrict__ parent_node,
                                                       int* __restrict__ parent_leaf, unsigned int* __restrict__ leaves) {
    const int m = *m_of, b0 = blockIdx.x * PLOC_P;
    if (m <= PLOC_TAIL) {
        if (blockIdx.x == 0 && threadIdx.x == 0) *m_next = m;
        return;
    }
    if (b0 >= m) return;
    constexpr int PER = PLOC_P / PLOC_T;
    int s = 0, p[PER];
    for (int b = threadIdx.x; b < (int)blockIdx.x; b += PLOC_T) s += gone[b];
    int mine = 0;
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        const int i = b0 + threadIdx.x * PER + k;
        p[k] = i < m ? pair[i] : -1;
        mine += p[k] >= 0 && p[k] < i;
    }
    int before, in_block;
    block_excl_scan<int, PLOC_T>(s, &before);
    int r = before + block_excl_scan<int, PLOC_T>(mine, &in_block);   // clusters gone before this thread's first
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        const int i = b0 + threadIdx.x * PER + k;
        if (i >= m) break;
        const bool up = p[k] >= 0 && p[k] < i;
        if (p[k] < 0) {
            blo2[i - r] = blo[i];
            bhi2[i - r] = bhi[i];
        } else if (up) {
            int between = 0;   // gone in [p, i)
            for (int y = p[k]; y < i; ++y) {
                const int py = pair[y];
                between += py >= 0 && py < y;
            }
            float4 al = blo[p[k]], ah = bhi[p[k]];
            ploc_node(m - 2 - r, al, ah, blo[i], bhi[i], nodes, parent_node, parent_leaf, leaves);
            const int to = p[k] - (r - between);
            blo2[to] = al;
            bhi2[to] = ah;
        }
        r += up;
        if (i == m - 1) *m_next = m - r;
    }
}

// The remaining rounds, PLOC_TAIL clusters or fewer, one block. m_of: the counts before each round
// launched so far; rounds alternate between the two cluster arrays until the first count of at most
// PLOC_TAIL. left: 1 when one cluster is left, more when no pair was mutual (non-finite boxes).
template <int R>
__global__ void __launch_bounds__(PLOC_TAIL) k_ploc_tail(const int* __restrict__ m_of, int rounds,
                                                         const float4* __restrict__ blo_a, const float4* __restrict__ bhi_a,
                                                         const float4* __restrict__ blo_b, const float4* __restrict__ bhi_b,
                                                         float4* __restrict__ nodes, int* __restrict__ parent_node,
                                                         int* __restrict__ parent_leaf, unsigned int* __restrict__ leaves,
                                                         int* __restrict__ left) {
    __shared__ float4 sl[PLOC_TAIL], sh[PLOC_TAIL];
    __shared__ int snn[PLOC_TAIL];
    __shared__ unsigned up_of[PLOC_TAIL / 32];
    __shared__ int gone_of[PLOC_TAIL / 32];
    int r0 = 0;
    while (r0 < rounds && m_of[r0] > PLOC_TAIL) ++r0;
    int m = m_of[r0];
    const int i = threadIdx.x, lane = i & 31, warp = i >> 5;
    if (m > PLOC_TAIL) {
        if (i == 0) *left = m;
        return;
    }
    float4 al = make_float4(0.f, 0.f, 0.f, 0.f), ah = al;
    if (i < m) {
        al = (r0 & 1 ? blo_b : blo_a)[i];
        ah = (r0 & 1 ? bhi_b : bhi_a)[i];
    }
    while (m > 1) {
        sl[i] = al;
        sh[i] = ah;
        __syncthreads();
        const int j = i < m ? ploc_nearest<R>(sl, sh, i, i, m) : -1;
        snn[i] = j;
        __syncthreads();
        const int p = j >= 0 && snn[j] == i ? j : -1;
        const bool up = p >= 0 && p < i;
        const unsigned mask = __ballot_sync(0xffffffffu, up);
        if (lane == 0) up_of[warp] = mask;
        __syncthreads();
        // clusters gone before each warp's first, and in all
        const int c = __popc(up_of[lane]);
        int incl = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int u = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += u;
        }
        if (warp == 0) gone_of[lane] = incl - c;
        const int all = __shfl_sync(0xffffffffu, incl, 31);
        const int mine = __shfl_sync(0xffffffffu, incl - c, warp);
        __syncthreads();
        if (all == 0) break;
        const int r = mine + __popc(mask & ((1u << lane) - 1u));
        int to = -1;
        float4 nl = al, nh = ah;
        if (i < m && p < 0) {
            to = i - r;
        } else if (up) {
            nl = sl[p];
            nh = sh[p];
            ploc_node(m - 2 - r, nl, nh, al, ah, nodes, parent_node, parent_leaf, leaves);
            to = p - (gone_of[p >> 5] + __popc(up_of[p >> 5] & ((1u << (p & 31)) - 1u)));
        }
        __syncthreads();   // every cluster has been read
        if (to >= 0) {
            sl[to] = nl;
            sh[to] = nh;
        }
        m -= all;
        __syncthreads();
        al = sl[i];
        ah = sh[i];
        __syncthreads();
    }
    if (i == 0) *left = m;
}

// ---- depth-first node layout ------------------------------------------------------------------
// Renumber the internal nodes in depth-first order (a node, then its left subtree, then its right
// subtree), so that a node's left child directly follows it in memory and often shares its
// cache line. leaves[v] = number of leaves below v (bottom-up); the index of v is the sum, over
// the path from the root, of 1 per step plus the left sibling's internal-node count when the
// step goes right.
// Leaves under every internal node, bottom-up: the second of a node's two children to arrive
// sums the children's counts and climbs on (one atomic per node, as in the box refit).
__global__ void k_leaf_counts(const int* __restrict__ parent_leaf, const int* __restrict__ parent_node,
                              const float4* __restrict__ nodes, int n, unsigned int* __restrict__ leaves,
                              unsigned int* __restrict__ flags) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    int p = parent_leaf[i];
    int guard = 0;
    while (p >= 0 && guard++ < 4096) {
        __threadfence();
        if (atomicAdd(&flags[p], 1u) == 0u) return;   // the sibling finishes this node
        __threadfence();
        const float4 l = nodes[4 * p + 3];
        const int a = __float_as_int(l.x), b = __float_as_int(l.y);
        const unsigned int ca = a >= 0 ? __ldcg(&leaves[a]) : 1u;
        const unsigned int cb = b >= 0 ? __ldcg(&leaves[b]) : 1u;
        leaves[p] = ca + cb;
        p = p > 0 ? parent_node[p] : -1;
    }
}

// even[index] = 1 where the node's depth is even (root 0): those become 4-wide nodes. *depth: the
// deepest leaf (one level below the deepest node), counted up to 4097; a tree above MAX_DEPTH is refused
// before anything reads dfs or even, which hold nothing for the nodes whose climb was cut off. left: the
// clusters that the clustering ended with (nullptr: another builder); without one root there is no tree.
constexpr unsigned MAX_DEPTH = 64;
__global__ void k_dfs_index(const float4* __restrict__ nodes, const int* __restrict__ parent_node,
                            const unsigned int* __restrict__ leaves, int n_int, const int* __restrict__ left,
                            int* __restrict__ dfs, int64_t* __restrict__ even, unsigned int* __restrict__ depth) {
    int v = blockIdx.x * blockDim.x + threadIdx.x;
    const unsigned live = __ballot_sync(0xffffffffu, v < n_int);
    if (v >= n_int || (left && *left != 1)) return;
    int idx = 0, u = v, steps = 0;
    while (u > 0 && steps < 4096) {
        ++steps;
        const int p = parent_node[u];
        const float4 l = nodes[4 * p + 3];
        const int left = __float_as_int(l.x);
        idx += 1;
        if (left != u) idx += left >= 0 ? (int)leaves[left] - 1 : 0;   // internal nodes of the left subtree
        u = p;
    }
    if (u <= 0) {
        dfs[v] = idx;
        even[idx] = (steps & 1) == 0 ? 1 : 0;
    }
    const unsigned deep = __reduce_max_sync(live, (unsigned)steps + 1u);
    if ((threadIdx.x & 31) == 0) atomicMax(depth, deep);
}

__global__ void k_dfs_remap(const float4* __restrict__ nodes, const int* __restrict__ dfs, int n_int,
                            float4* __restrict__ out) {
    int v = blockIdx.x * blockDim.x + threadIdx.x;
    if (v >= n_int) return;
    const int d = dfs[v];
    out[4 * d + 0] = nodes[4 * v + 0];
    out[4 * d + 1] = nodes[4 * v + 1];
    out[4 * d + 2] = nodes[4 * v + 2];
    const float4 l = nodes[4 * v + 3];
    const int a = __float_as_int(l.x), b = __float_as_int(l.y);
    out[4 * d + 3] = make_float4(__int_as_float(a >= 0 ? dfs[a] : a), __int_as_float(b >= 0 ? dfs[b] : b), 0.f, 0.f);
}

// ---- dynamic scenes: re-pose every mesh, refit the boxes over the unchanged topology ----------
// Mesh-local triangle vertices in stored (mesh) order, kept for re-posing.
__global__ void k_gather_local(const float* __restrict__ v, const uint32_t* __restrict__ idx, uint32_t nt,
                               uint32_t nv, uint32_t tri_base, float4* __restrict__ tri_local) {
    uint32_t t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= nt) return;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        uint32_t vi = idx[3 * t + k];
        if (vi >= nv) vi = 0;   // the world gather of the same mesh reports the bad index
        tri_local[3 * (tri_base + t) + k] = make_float4(v[3 * vi], v[3 * vi + 1], v[3 * vi + 2], 0.f);
    }
}

// World triangles of a new pose: the transform of k_transform (same FP64 operation order, so a
// pose equal to the build's transforms reproduces the built triangles bit for bit), one thread
// per triangle; scene bounds as in k_gather (centroid box in [0, 6), vertex box in [6, 12)).
__global__ void k_pose(const float4* __restrict__ tri_local, const uint32_t* __restrict__ tri_mesh,
                       const double* __restrict__ xf, uint32_t nt, float4* __restrict__ tri_canon,
                       unsigned int* __restrict__ bounds) {
    uint32_t t = blockIdx.x * blockDim.x + threadIdx.x;
    float lo[6], hi[6];
#pragma unroll
    for (int c = 0; c < 6; ++c) { lo[c] = INFINITY; hi[c] = -INFINITY; }
    if (t < nt) {
        const double* M = xf + 12 * tri_mesh[t];
        float w[9];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const float4 p = tri_local[3 * t + k];
            const double x = p.x, y = p.y, z = p.z;
#pragma unroll
            for (int r = 0; r < 3; ++r) {
                double a = __dadd_rn(__dmul_rn(M[4 * r + 0], x), __dmul_rn(M[4 * r + 1], y));
                a = __dadd_rn(a, __dmul_rn(M[4 * r + 2], z));
                a = __dadd_rn(a, M[4 * r + 3]);
                w[3 * k + r] = __double2float_rn(a);
            }
            tri_canon[3 * t + k] = make_float4(w[3 * k], w[3 * k + 1], w[3 * k + 2], 0.f);
        }
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            lo[a] = hi[a] = (w[a] + w[3 + a] + w[6 + a]) * (1.f / 3.f);
            lo[3 + a] = fminf(fminf(w[a], w[3 + a]), w[6 + a]);
            hi[3 + a] = fmaxf(fmaxf(w[a], w[3 + a]), w[6 + a]);
        }
    }
    fold_bounds(lo, hi, bounds);
}

// Triangle id of every leaf slot (v0.w of the leaf-order copy).
__global__ void k_leaf_order(const float4* __restrict__ bvh_tris, uint32_t n, uint32_t* __restrict__ order) {
    uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) order[i] = __float_as_uint(bvh_tris[3 * i].w);
}

// Parents in the final node layout, from the child links (root: -1 from the memset).
__global__ void k_final_parents(const float4* __restrict__ nodes, int n_int, int n_leaves,
                                int* __restrict__ parent_node, int* __restrict__ parent_leaf) {
    int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= n_int) return;
    const float4 l = nodes[4 * p + 3];
    const int c[2] = {__float_as_int(l.x), __float_as_int(l.y)};
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        if (c[k] >= 0) {
            if (c[k] < n_int) parent_node[c[k]] = p;
        } else if (~c[k] < n_leaves) {
            parent_leaf[~c[k]] = p;
        }
    }
}

}  // namespace

// Inverse affine maps (world -> mesh-local, row-major 3 x 4) of row-major 4 x 4 transforms, by the
// adjugate in FP64; false if any transform is singular (its rows are left zero).
static bool mesh_inverses(const double* xf, uint32_t n_meshes, std::vector<double>& inv) {
    inv.assign(12 * (size_t)n_meshes, 0.0);
    bool ok = true;
    for (uint32_t m = 0; m < n_meshes; ++m) {
        const double* M = xf + 16 * m;
        const double a = M[0], b = M[1], c = M[2], d = M[4], e2 = M[5], f = M[6], g = M[8], h = M[9], k = M[10];
        const double det = a * (e2 * k - f * h) - b * (d * k - f * g) + c * (d * h - e2 * g);
        if (!(std::fabs(det) > 1e-300) || !std::isfinite(det)) {
            ok = false;
            continue;
        }
        const double r[9] = {(e2 * k - f * h) / det, (c * h - b * k) / det, (b * f - c * e2) / det,
                             (f * g - d * k) / det,  (a * k - c * g) / det,  (c * d - a * f) / det,
                             (d * h - e2 * g) / det, (b * g - a * h) / det,  (a * e2 - b * d) / det};
        for (int i = 0; i < 3; ++i) {
            for (int j = 0; j < 3; ++j) inv[12 * m + 4 * i + j] = r[3 * i + j];
            inv[12 * m + 4 * i + 3] = -(r[3 * i] * M[3] + r[3 * i + 1] * M[7] + r[3 * i + 2] * M[11]);
        }
    }
    return ok;
}

static gm_status build_scene(gm_ctx* ctx, const gm_mesh_desc* meshes, uint32_t n_meshes, int builder,
                             bool dynamic, int ploc_radius, gm_stream stream, gm_scene** out) {
    if (!ctx || !meshes || !out || n_meshes == 0)
        return gm_set_error(GM_ERR_INVALID_ARG, "gm_build_scene: null argument or no meshes");
    *out = nullptr;
    cudaStream_t s = (cudaStream_t)stream;
    uint64_t nt64 = 0;
    for (uint32_t m = 0; m < n_meshes; ++m) {
        const gm_mesh_desc& d = meshes[m];
        if (d.n_tris > 0 && (!d.vertices || !d.indices || d.n_verts == 0))
            return gm_set_error(GM_ERR_INVALID_ARG, "gm_build_scene: mesh " + std::to_string(m) + " has triangles but no vertices/indices");
        for (int k = 0; k < 16; ++k)
            if (!std::isfinite(d.transform[k]))
                return gm_set_error(GM_ERR_INVALID_ARG, "gm_build_scene: non-finite transform");
        nt64 += d.n_tris;
    }
    if (nt64 == 0) return gm_set_error(GM_ERR_INVALID_ARG, "gm_build_scene: the scene has no triangles");
    if (nt64 > 0x7fffffffu) return gm_set_error(GM_ERR_UNSUPPORTED, "gm_build_scene: more than 2^31-1 triangles");
    GM_TRY_CUDA(cudaSetDevice(ctx->device));
    const uint32_t nt = (uint32_t)nt64;

    gm_scene* sc = new gm_scene();
    sc->ctx = ctx;
    sc->n_tris = nt;
    sc->n_meshes = n_meshes;
    std::vector<void*> tmp;
    auto fail = [&](gm_status st) {
        for (void* p : tmp) cudaFreeAsync(p, s);
        gm_scene_free(sc);
        return st;
    };
    gm_status st;
#define SC_ALLOC(ptr, bytes) \
    if ((st = gm_alloc((void**)&(ptr), (bytes), s)) != GM_OK) return fail(st)
#define TMP_ALLOC(ptr, bytes)                                          \
    do {                                                               \
        if ((st = gm_alloc((void**)&(ptr), (bytes), s)) != GM_OK) return fail(st); \
        tmp.push_back((void*)(ptr));                                   \
    } while (0)

    SC_ALLOC(sc->tri_canon, sizeof(float4) * 3 * (size_t)nt);
    SC_ALLOC(sc->tri_mesh, sizeof(uint32_t) * (size_t)nt);
    SC_ALLOC(sc->mesh_object, sizeof(uint32_t) * n_meshes);
    SC_ALLOC(sc->bvh_tris, sizeof(float4) * 3 * (size_t)nt);
    if (dynamic) SC_ALLOC(sc->tri_local, sizeof(float4) * 3 * (size_t)nt);
    if (nt > 1) SC_ALLOC(sc->nodes, sizeof(float4) * 4 * (size_t)(nt - 1));
    unsigned int* bounds = nullptr;
    int* err = nullptr;
    TMP_ALLOC(bounds, sizeof(unsigned int) * 16);
    err = ctx->dev_err;
    k_bounds_init<<<1, 32, 0, s>>>(bounds);
    int launches = 1;

    std::vector<uint32_t> objs(n_meshes);
    uint32_t base = 0;
    for (uint32_t m = 0; m < n_meshes; ++m) {
        const gm_mesh_desc& d = meshes[m];
        objs[m] = d.object_id;
        if (d.n_tris == 0) continue;
        void *dv = nullptr, *di = nullptr;
        bool ov = false, oi = false;
        if ((st = gm_stage_to_device(d.vertices, sizeof(float) * 3 * (size_t)d.n_verts, s, &dv, &ov)) != GM_OK) return fail(st);
        if (ov) tmp.push_back(dv);
        if ((st = gm_stage_to_device(d.indices, sizeof(uint32_t) * 3 * (size_t)d.n_tris, s, &di, &oi)) != GM_OK) return fail(st);
        if (oi) tmp.push_back(di);
        float* wv = nullptr;
        TMP_ALLOC(wv, sizeof(float) * 3 * (size_t)d.n_verts);
        Mat16 M;
        memcpy(M.m, d.transform, sizeof(M.m));
        k_transform<<<gm_div_up(d.n_verts, 256), 256, 0, s>>>((const float*)dv, d.n_verts, M, wv);
        k_gather<<<gm_div_up(d.n_tris, 256), 256, 0, s>>>(wv, (const uint32_t*)di, d.n_tris, d.n_verts, base, m,
                                                          sc->tri_canon, sc->tri_mesh, bounds, err);
        launches += 2;
        if (dynamic) {
            k_gather_local<<<gm_div_up(d.n_tris, 256), 256, 0, s>>>((const float*)dv, (const uint32_t*)di, d.n_tris,
                                                                    d.n_verts, base, sc->tri_local);
            ++launches;
        }
        base += d.n_tris;
    }
    cudaError_t ce = cudaMemcpyAsync(sc->mesh_object, objs.data(), sizeof(uint32_t) * n_meshes, cudaMemcpyHostToDevice, s);
    auto wait_fail = [&](gm_status st_) {   // host temporaries may still be read
        cudaStreamSynchronize(s);
        return fail(st_);
    };
    if (ce != cudaSuccess) return wait_fail(gm_cuda_error(ce, "gm_build_scene"));
    // world -> mesh-local maps for the export format (affine inverse in FP64); the host copies live until
    // the stream is waited for below
    std::vector<double> xf(16 * (size_t)n_meshes), inv;
    for (uint32_t m = 0; m < n_meshes; ++m) memcpy(&xf[16 * m], meshes[m].transform, sizeof(double) * 16);
    sc->mesh_inv_ok = mesh_inverses(xf.data(), n_meshes, inv);
    SC_ALLOC(sc->mesh_inv, sizeof(double) * 12 * n_meshes);
    if ((ce = cudaMemcpyAsync(sc->mesh_inv, inv.data(), sizeof(double) * 12 * n_meshes, cudaMemcpyHostToDevice, s)) !=
        cudaSuccess)
        return wait_fail(gm_cuda_error(ce, "gm_build_scene"));

    uint64_t* keys = nullptr;
    uint32_t* order = nullptr;
    int *parent_node = nullptr, *parent_leaf = nullptr;
    unsigned int *leaves = nullptr, *depth = nullptr;
    const uint32_t n_in = nt > 1 ? nt - 1 : 1;
    TMP_ALLOC(keys, sizeof(uint64_t) * nt);
    TMP_ALLOC(order, sizeof(uint32_t) * nt);
    TMP_ALLOC(parent_leaf, sizeof(int) * nt);
    TMP_ALLOC(parent_node, sizeof(int) * n_in);
    TMP_ALLOC(leaves, sizeof(unsigned int) * n_in);
    TMP_ALLOC(depth, sizeof(unsigned int) * 2);   // [0] depth, [1] clusters left
    // -1 everywhere: a link the hierarchy step did not write stops the refit instead of escaping
    if ((ce = cudaMemsetAsync(parent_leaf, 0xff, sizeof(int) * nt, s)) != cudaSuccess ||
        (ce = cudaMemsetAsync(parent_node, 0xff, sizeof(int) * n_in, s)) != cudaSuccess ||
        (ce = cudaMemsetAsync(depth, 0, sizeof(unsigned int) * 2, s)) != cudaSuccess)
        return wait_fail(gm_cuda_error(ce, "gm_build_scene"));
    k_morton<<<gm_div_up(nt, 256), 256, 0, s>>>(sc->tri_canon, nt, bounds, keys, order);
    ++launches;
    if ((st = gm_radix_sort_u64(keys, order, nt, 63, s, &launches)) != GM_OK) return wait_fail(st);
    const bool ploc = builder == GM_BUILD_PLOC && nt > 1;
    bool cut = false;   // the clustering was still merging after its last round
    if (ploc) {
        constexpr int kRounds = 4096;
        int *m_of = nullptr, *pair = nullptr, *gone = nullptr;
        float4 *lo[2] = {}, *hi[2] = {};
        const uint32_t nblk = gm_div_up(nt, PLOC_P);
        TMP_ALLOC(m_of, sizeof(int) * (kRounds + PLOC_BATCH + 1));
        for (int k = 0; k < 2; ++k) {
            TMP_ALLOC(lo[k], sizeof(float4) * nt);
            TMP_ALLOC(hi[k], sizeof(float4) * nt);
        }
        TMP_ALLOC(pair, sizeof(int) * nt);
        TMP_ALLOC(gone, sizeof(int) * nblk);
        k_ploc_init<<<gm_div_up(nt, 256), 256, 0, s>>>(sc->tri_canon, order, (int)nt, bounds, lo[0], hi[0], sc->bvh_tris,
                                                       m_of);
        ++launches;
        int m = (int)nt, rounds = 0;
        while (m > PLOC_TAIL && rounds < kRounds) {
            const uint32_t grid = gm_div_up((uint32_t)m, PLOC_P);
            for (int k = 0; k < PLOC_BATCH; ++k, ++rounds) {
                const int a = rounds & 1;
                switch (ploc_radius) {
                    case 4: k_ploc_pair<4><<<grid, PLOC_T, 0, s>>>(m_of + rounds, lo[a], hi[a], pair, gone); break;
                    case 16: k_ploc_pair<16><<<grid, PLOC_T, 0, s>>>(m_of + rounds, lo[a], hi[a], pair, gone); break;
                    case 32: k_ploc_pair<32><<<grid, PLOC_T, 0, s>>>(m_of + rounds, lo[a], hi[a], pair, gone); break;
                    case 64: k_ploc_pair<64><<<grid, PLOC_T, 0, s>>>(m_of + rounds, lo[a], hi[a], pair, gone); break;
                    default: k_ploc_pair<8><<<grid, PLOC_T, 0, s>>>(m_of + rounds, lo[a], hi[a], pair, gone); break;
                }
                k_ploc_apply<<<grid, PLOC_T, 0, s>>>(m_of + rounds, m_of + rounds + 1, lo[a], hi[a], pair, gone,
                                                     lo[a ^ 1], hi[a ^ 1], sc->nodes, parent_node, parent_leaf, leaves);
            }
            launches += 2 * PLOC_BATCH;
            int now = 0;
            if ((ce = cudaMemcpyAsync(&now, m_of + rounds, sizeof(int), cudaMemcpyDeviceToHost, s)) != cudaSuccess ||
                (ce = cudaStreamSynchronize(s)) != cudaSuccess)
                return wait_fail(gm_cuda_error(ce, "gm_build_scene (clustering)"));
            if (now >= m) break;   // no mutual pair: reported below
            m = now;
            cut = m > PLOC_TAIL && rounds >= kRounds;
        }
        auto tail = [&](auto kern) {
            kern<<<1, PLOC_TAIL, 0, s>>>(m_of, rounds, lo[0], hi[0], lo[1], hi[1], sc->nodes, parent_node, parent_leaf,
                                         leaves, (int*)depth + 1);
        };
        switch (ploc_radius) {
            case 4: tail(k_ploc_tail<4>); break;
            case 16: tail(k_ploc_tail<16>); break;
            case 32: tail(k_ploc_tail<32>); break;
            case 64: tail(k_ploc_tail<64>); break;
            default: tail(k_ploc_tail<8>); break;
        }
        ++launches;
    } else {
        unsigned int* flags = nullptr;
        TMP_ALLOC(flags, sizeof(unsigned int) * n_in);
        if ((ce = cudaMemsetAsync(flags, 0, sizeof(unsigned int) * n_in, s)) != cudaSuccess)
            return wait_fail(gm_cuda_error(ce, "gm_build_scene"));
        if (nt > 1) k_hierarchy<<<gm_div_up(nt - 1, 256), 256, 0, s>>>(keys, (int)nt, sc->nodes, parent_node, parent_leaf);
        k_refit<<<gm_div_up(nt, 256), 256, 0, s>>>(sc->tri_canon, order, (int)nt, sc->nodes, parent_node, parent_leaf,
                                                    flags, bounds, sc->bvh_tris);
        launches += (nt > 1 ? 2 : 1);
    }
    int* dfs = nullptr;
    int64_t* incl = nullptr;
    const int n_int = (int)nt - 1;
    if (nt > 1) {
        TMP_ALLOC(dfs, sizeof(int) * n_int);
        if (dynamic) {
            SC_ALLOC(sc->incl4, sizeof(int64_t) * n_int);
            incl = sc->incl4;
        } else {
            TMP_ALLOC(incl, sizeof(int64_t) * n_int);
        }
        if (!ploc) {   // the clustering counted the leaves as it merged
            unsigned int* arrived = nullptr;
            TMP_ALLOC(arrived, sizeof(unsigned int) * n_int);
            if ((ce = cudaMemsetAsync(leaves, 0, sizeof(unsigned int) * n_int, s)) != cudaSuccess ||
                (ce = cudaMemsetAsync(arrived, 0, sizeof(unsigned int) * n_int, s)) != cudaSuccess)
                return wait_fail(gm_cuda_error(ce, "gm_build_scene"));
            k_leaf_counts<<<gm_div_up(nt, 256), 256, 0, s>>>(parent_leaf, parent_node, sc->nodes, (int)nt, leaves, arrived);
            ++launches;
        }
        k_dfs_index<<<gm_div_up(n_int, 256), 256, 0, s>>>(sc->nodes, parent_node, leaves, n_int,
                                                          ploc ? (int*)depth + 1 : nullptr, dfs, incl, depth);
        ++launches;
    }
    ctx->launches += launches;
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return wait_fail(gm_cuda_error(e, "gm_build_scene launch"));
    unsigned int hb[16] = {0};
    unsigned int hdepth[2] = {0, 0};
    int herr = 0;
    if ((e = cudaMemcpyAsync(hb, bounds, sizeof(unsigned int) * 12, cudaMemcpyDeviceToHost, s)) != cudaSuccess ||
        (e = cudaMemcpyAsync(hdepth, depth, sizeof(hdepth), cudaMemcpyDeviceToHost, s)) != cudaSuccess ||
        (e = cudaMemcpyAsync(&herr, err, sizeof(int), cudaMemcpyDeviceToHost, s)) != cudaSuccess ||
        (e = cudaStreamSynchronize(s)) != cudaSuccess)
        return wait_fail(gm_cuda_error(e, "gm_build_scene"));
    if (herr == GM_DEV_BAD_INDEX) {
        cudaMemsetAsync(ctx->dev_err, 0, sizeof(int), s);
        return fail(gm_set_error(GM_ERR_INVALID_ARG, "gm_build_scene: a vertex index is out of range"));
    }
    if (cut)   // one pair a round, as runs of equal boxes merge: a chain
        return fail(gm_set_error(GM_ERR_UNSUPPORTED, "gm_build_scene: BVH deeper than 64 levels (" + std::to_string(hdepth[1]) +
                                                         " clusters left after 4096 rounds)"));
    if (ploc && hdepth[1] != 1)   // no mutual pair: cannot happen with consistent tie-breaking and finite boxes
        return fail(gm_set_error(GM_ERR_INTERNAL, "gm_build_scene: clustering made no progress"));
    auto dec = [](unsigned int o) {
        unsigned int b = (o & 0x80000000u) ? (o & 0x7fffffffu) : ~o;
        float f;
        memcpy(&f, &b, 4);
        return f;
    };
    for (int k = 0; k < 3; ++k) {
        sc->box_lo[k] = dec(hb[6 + k]);
        sc->box_hi[k] = dec(hb[9 + k]);
        if (!std::isfinite(sc->box_lo[k]) || !std::isfinite(sc->box_hi[k]))
            return fail(gm_set_error(GM_ERR_INVALID_ARG, "gm_build_scene: non-finite vertex"));
    }
    // the layout below uses the depth: nothing of a deeper tree is laid out
    sc->depth = nt > 1 ? hdepth[0] : 0;
    if (sc->depth > MAX_DEPTH)
        return fail(gm_set_error(GM_ERR_UNSUPPORTED, "gm_build_scene: BVH deeper than 64 levels (" +
                                                         std::to_string(sc->depth) + ")"));
    if (nt > 1) {
        float4* reordered = nullptr;
        launches = 1;
        if ((st = gm_alloc((void**)&reordered, sizeof(float4) * 4 * (size_t)n_int, s)) != GM_OK) return fail(st);
        k_dfs_remap<<<gm_div_up(n_int, 256), 256, 0, s>>>(sc->nodes, dfs, n_int, reordered);
        cudaFreeAsync(sc->nodes, s);
        sc->nodes = reordered;
        // the 4-wide nodes follow the depth-first order. Every even-depth node but the root is a child of
        // an odd-depth one, so at most (2 n_int + 1) / 3 of the nodes are of even depth.
        if ((st = gm_inclusive_scan_i64(incl, (uint32_t)n_int, s, &launches)) != GM_OK) return fail(st);
        SC_ALLOC(sc->nodes4, sizeof(float4) * 8 * ((2 * (size_t)n_int + 1) / 3));
        k_collapse4<<<gm_div_up(n_int, 256), 256, 0, s>>>(sc->nodes, n_int, incl, sc->nodes4);
        ++launches;
        ctx->launches += launches;
        if ((e = cudaGetLastError()) != cudaSuccess || (e = cudaStreamSynchronize(s)) != cudaSuccess)
            return wait_fail(gm_cuda_error(e, "gm_build_scene layout"));
    }
    for (void* p : tmp) cudaFreeAsync(p, s);
    tmp.clear();
    *out = sc;
    return GM_OK;
#undef SC_ALLOC
#undef TMP_ALLOC
}

extern "C" gm_status gm_build_scene(gm_ctx* ctx, const gm_mesh_desc* meshes, uint32_t n_meshes, gm_stream stream,
                                    gm_scene** out) {
    return build_scene(ctx, meshes, n_meshes, GM_BUILD_DEFAULT, false, kPlocRadius, stream, out);
}

extern "C" gm_status gm_build_scene_opts(gm_ctx* ctx, const gm_mesh_desc* meshes, uint32_t n_meshes,
                                         const gm_build_opts* opts, gm_stream stream, gm_scene** out) {
    const int b = opts ? opts->builder : GM_BUILD_DEFAULT;
    if (b != GM_BUILD_LBVH && b != GM_BUILD_PLOC)
        return gm_set_error(GM_ERR_INVALID_ARG, "gm_build_scene_opts: unknown builder");
    const int r = opts && opts->ploc_radius ? opts->ploc_radius : kPlocRadius;
    if (r != 4 && r != 8 && r != 16 && r != 32 && r != 64)
        return gm_set_error(GM_ERR_INVALID_ARG, "gm_build_scene_opts: ploc_radius must be 4, 8, 16, 32 or 64");
    return build_scene(ctx, meshes, n_meshes, b, opts && opts->dynamic != 0, r, stream, out);
}

extern "C" gm_status gm_scene_pose(gm_scene* sc, const double* transforms, gm_stream stream) {
    if (!sc || !transforms) return gm_set_error(GM_ERR_INVALID_ARG, "gm_scene_pose: null argument");
    if (!sc->tri_local)
        return gm_set_error(GM_ERR_INVALID_ARG, "gm_scene_pose: the scene was not built with gm_build_opts.dynamic");
    const uint32_t nm = sc->n_meshes, nt = sc->n_tris;
    for (size_t k = 0; k < 16 * (size_t)nm; ++k)
        if (!std::isfinite(transforms[k])) return gm_set_error(GM_ERR_INVALID_ARG, "gm_scene_pose: non-finite transform");
    cudaStream_t s = (cudaStream_t)stream;
    gm_ctx* ctx = sc->ctx;
    GM_TRY_CUDA(cudaSetDevice(ctx->device));
    std::vector<double> xf12(12 * (size_t)nm);
    for (uint32_t m = 0; m < nm; ++m) memcpy(&xf12[12 * m], transforms + 16 * m, sizeof(double) * 12);
    std::vector<double> inv;
    const bool inv_ok = mesh_inverses(transforms, nm, inv);
    std::vector<void*> tmp;
    auto done = [&](gm_status st) {
        for (void* p : tmp) cudaFreeAsync(p, s);
        return st;
    };
    gm_status st;
#define POSE_TMP(ptr, bytes)                                                          \
    do {                                                                              \
        if ((st = gm_alloc((void**)&(ptr), (bytes), s)) != GM_OK) return done(st);    \
        tmp.push_back((void*)(ptr));                                                  \
    } while (0)
    double* d_xf = nullptr;
    unsigned int* bounds = nullptr;
    uint32_t* order = nullptr;
    int *parent_node = nullptr, *parent_leaf = nullptr;
    unsigned int* flags = nullptr;
    const uint32_t n_int = nt > 1 ? nt - 1 : 1;
    POSE_TMP(d_xf, sizeof(double) * 12 * nm);
    POSE_TMP(bounds, sizeof(unsigned int) * 16);
    POSE_TMP(order, sizeof(uint32_t) * nt);
    POSE_TMP(parent_node, sizeof(int) * n_int);
    POSE_TMP(parent_leaf, sizeof(int) * nt);
    POSE_TMP(flags, sizeof(unsigned int) * n_int);
#undef POSE_TMP
    cudaError_t e;
    if ((e = cudaMemcpyAsync(d_xf, xf12.data(), sizeof(double) * 12 * nm, cudaMemcpyHostToDevice, s)) != cudaSuccess ||
        (e = cudaMemcpyAsync(sc->mesh_inv, inv.data(), sizeof(double) * 12 * nm, cudaMemcpyHostToDevice, s)) != cudaSuccess ||
        (e = cudaMemsetAsync(parent_node, 0xff, sizeof(int) * n_int, s)) != cudaSuccess ||
        (e = cudaMemsetAsync(parent_leaf, 0xff, sizeof(int) * nt, s)) != cudaSuccess ||
        (e = cudaMemsetAsync(flags, 0, sizeof(unsigned int) * n_int, s)) != cudaSuccess)
        return done(gm_cuda_error(e, "gm_scene_pose"));
    k_bounds_init<<<1, 32, 0, s>>>(bounds);
    k_pose<<<gm_div_up(nt, 256), 256, 0, s>>>(sc->tri_local, sc->tri_mesh, d_xf, nt, sc->tri_canon, bounds);
    k_leaf_order<<<gm_div_up(nt, 256), 256, 0, s>>>(sc->bvh_tris, nt, order);
    int launches = 3;
    if (nt > 1) {
        k_final_parents<<<gm_div_up(nt - 1, 256), 256, 0, s>>>(sc->nodes, (int)(nt - 1), (int)nt, parent_node,
                                                               parent_leaf);
        ++launches;
    }
    // leaf-order triangles rewritten from the posed ones, then the boxes bottom-up (the
    // hierarchy and its depth are unchanged)
    k_refit<<<gm_div_up(nt, 256), 256, 0, s>>>(sc->tri_canon, order, (int)nt, sc->nodes, parent_node, parent_leaf,
                                                flags, bounds, sc->bvh_tris);
    ++launches;
    if (nt > 1) {   // the 4-wide nodes take the new boxes
        k_collapse4<<<gm_div_up(nt - 1, 256), 256, 0, s>>>(sc->nodes, (int)(nt - 1), sc->incl4, sc->nodes4);
        ++launches;
    }
    unsigned int hb[12] = {0};
    if ((e = cudaGetLastError()) != cudaSuccess ||
        (e = cudaMemcpyAsync(hb, bounds, sizeof(hb), cudaMemcpyDeviceToHost, s)) != cudaSuccess ||
        (e = cudaStreamSynchronize(s)) != cudaSuccess)
        return done(gm_cuda_error(e, "gm_scene_pose"));
    ctx->launches += launches;
    auto dec = [](unsigned int o) {
        unsigned int b = (o & 0x80000000u) ? (o & 0x7fffffffu) : ~o;
        float f;
        memcpy(&f, &b, 4);
        return f;
    };
    for (int k = 0; k < 3; ++k) {
        sc->box_lo[k] = dec(hb[6 + k]);
        sc->box_hi[k] = dec(hb[9 + k]);
    }
    sc->mesh_inv_ok = inv_ok;
    for (int k = 0; k < 3; ++k)
        if (!std::isfinite(sc->box_lo[k]) || !std::isfinite(sc->box_hi[k]))
            return done(gm_set_error(GM_ERR_INVALID_ARG, "gm_scene_pose: non-finite vertex"));
    return done(GM_OK);
}

extern "C" gm_status gm_scene_info(const gm_scene* sc, uint32_t* n_tris, uint32_t* bvh_depth) {
    if (!sc) return gm_set_error(GM_ERR_INVALID_ARG, "gm_scene_info: null scene");
    if (n_tris) *n_tris = sc->n_tris;
    if (bvh_depth) *bvh_depth = sc->depth;
    return GM_OK;
}

namespace {
__global__ void k_unpack_tris(const float4* __restrict__ t, uint32_t nt, float* __restrict__ out) {
    uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nt) return;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        float4 v = t[3 * i + k];
        out[9 * i + 3 * k + 0] = v.x;
        out[9 * i + 3 * k + 1] = v.y;
        out[9 * i + 3 * k + 2] = v.z;
    }
}
}  // namespace

extern "C" gm_status gm_scene_triangles(const gm_scene* sc, float* dst, gm_stream stream) {
    if (!sc || !dst) return gm_set_error(GM_ERR_INVALID_ARG, "gm_scene_triangles: null argument");
    cudaStream_t s = (cudaStream_t)stream;
    size_t bytes = sizeof(float) * 9 * (size_t)sc->n_tris;
    bool dev = gm_is_device_ptr(dst);
    float* tmp = dst;
    if (!dev) GM_TRY(gm_alloc((void**)&tmp, bytes, s));
    k_unpack_tris<<<gm_div_up(sc->n_tris, 256), 256, 0, s>>>(sc->tri_canon, sc->n_tris, tmp);
    sc->ctx->launches += 1;
    if (!dev) {
        gm_status st = gm_copy_out(dst, tmp, bytes, s);
        cudaFreeAsync(tmp, s);
        return st;
    }
    GM_TRY_CUDA(cudaGetLastError());
    return GM_OK;
}

extern "C" void gm_scene_free(gm_scene* sc) {
    if (!sc) return;
    cudaFree(sc->tri_canon);
    cudaFree(sc->tri_mesh);
    cudaFree(sc->mesh_object);
    cudaFree(sc->mesh_inv);
    cudaFree(sc->nodes);
    cudaFree(sc->nodes4);
    cudaFree(sc->incl4);
    cudaFree(sc->bvh_tris);
    cudaFree(sc->tri_local);
    delete sc;
}
