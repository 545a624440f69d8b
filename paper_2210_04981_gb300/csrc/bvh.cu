// Acceleration structure standing in for the paper's hardware ray-tracing
// acceleration (Abstract), plus the closest-hit query used to check it.
//
// Common steps: scene and centroid bounds -> 63-bit Morton codes -> radix
// sort of (code, triangle) pairs -> triangles, materials and UVs stored in
// sorted order.  The hierarchy over the sorted triangles is then built by
// PLOC (parallel locally-ordered clustering, Meister and Bittner 2018; the
// default, HDOF_BUILDER=1) or by the linear BVH of Karras ("Maximizing
// parallelism in the construction of BVHs, octrees and k-d trees", HPG 2012;
// HDOF_BUILDER=0): one thread per internal node finds its key range and
// split, one thread per leaf refits child boxes bottom-up.  On the 1080p room
// the clustered tree needs 64 node visits per thin-lens ray against 100 for
// the linear one (2.5 ms against 3.3 ms for the frame's 3.4M rays).
#include <cub/cub.cuh>

#include <algorithm>
#include <cmath>
#include <cstring>

#include "internal.h"

namespace hdof {
namespace {

__device__ __forceinline__ unsigned f2ord(float f) {
    unsigned u = __float_as_uint(f);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float ord2f(unsigned u) {
    return __uint_as_float((u & 0x80000000u) ? (u & 0x7fffffffu) : ~u);
}

// bounds[0..5]: ordered-float vertex bounds of the scene (lo xyz, hi xyz);
// [6]: bad-index flag; [7]: number of scene-sized triangles;
// [8..13]: centroid bounds of the other triangles; [14..19]: centroid bounds of all
constexpr int NB = 20;

// Vertex bounds, the centroid bounds of all triangles and the bad-index flag.
// Reduced per block first: the warps' atomics on a dozen addresses were the
// kernel's time.
__global__ void __launch_bounds__(256) k_scene_bounds(const float* __restrict__ v, int nv, const int* __restrict__ idx,
                                                      int n, unsigned* bounds) {
    const float BIG = 3.4e38f;
    float x[12];  // vertex lo, hi, centroid lo, hi
#pragma unroll
    for (int k = 0; k < 12; ++k) x[k] = (k / 3) & 1 ? -BIG : BIG;
    bool bad = false;
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < n; t += gridDim.x * blockDim.x) {
        int a = idx[3 * t], b = idx[3 * t + 1], c = idx[3 * t + 2];
        if (a < 0 || b < 0 || c < 0 || a >= nv || b >= nv || c >= nv) {
            bad = true;
            continue;
        }
        for (int k = 0; k < 3; ++k) {
            const float p = v[3 * a + k], q = v[3 * b + k], r = v[3 * c + k], cen = (p + q + r) * (1.f / 3.f);
            x[k] = fminf(x[k], fminf(p, fminf(q, r)));
            x[3 + k] = fmaxf(x[3 + k], fmaxf(p, fmaxf(q, r)));
            x[6 + k] = fminf(x[6 + k], cen);
            x[9 + k] = fmaxf(x[9 + k], cen);
        }
    }
    __shared__ float red[8][12];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < 12; ++k) {
        const bool mx = (k / 3) & 1;
        for (int o = 16; o; o >>= 1) {
            const float y = __shfl_xor_sync(0xffffffffu, x[k], o);
            x[k] = mx ? fmaxf(x[k], y) : fminf(x[k], y);
        }
        if (lane == 0) red[w][k] = x[k];
    }
    const bool any_bad = __syncthreads_or(bad);
    if (threadIdx.x < 12) {
        const int k = threadIdx.x;
        const bool mx = (k / 3) & 1;
        float y = red[0][k];
        for (int j = 1; j < 8; ++j) y = mx ? fmaxf(y, red[j][k]) : fminf(y, red[j][k]);
        unsigned* dst = &bounds[k < 6 ? k : 14 + k - 6];
        if (mx) atomicMax(dst, f2ord(y));
        else atomicMin(dst, f2ord(y));
    }
    if (threadIdx.x == 0 && any_bad) atomicOr(&bounds[6], 1u);
}

__device__ __forceinline__ float box_area(const float lo[3], const float hi[3]) {
    float x = hi[0] - lo[0], y = hi[1] - lo[1], z = hi[2] - lo[2];
    return 2.f * (x * y + y * z + z * x);
}

// A triangle whose box covers more than big_frac of the scene box's surface
// area is "scene-sized" (room walls): kept out of the tree, where its box
// would widen every ancestor, and tested by every ray instead.
__global__ void k_classify(const float* __restrict__ v, const int* __restrict__ idx, int n, float big_frac,
                           unsigned* bounds, uint8_t* big) {
    float slo[3], shi[3];
    for (int k = 0; k < 3; ++k) {
        slo[k] = ord2f(bounds[k]);
        shi[k] = ord2f(bounds[3 + k]);
    }
    const float thr = big_frac * box_area(slo, shi);
    float lo[3] = {3.4e38f, 3.4e38f, 3.4e38f}, hi[3] = {-3.4e38f, -3.4e38f, -3.4e38f};
    unsigned nbig = 0;
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < n; t += gridDim.x * blockDim.x) {
        int a = idx[3 * t], b = idx[3 * t + 1], c = idx[3 * t + 2];
        float tlo[3], thi[3], cen[3];
        for (int k = 0; k < 3; ++k) {
            float x = v[3 * a + k], y = v[3 * b + k], z = v[3 * c + k];
            tlo[k] = fminf(x, fminf(y, z));
            thi[k] = fmaxf(x, fmaxf(y, z));
            cen[k] = (x + y + z) * (1.f / 3.f);
        }
        bool is_big = box_area(tlo, thi) > thr;
        big[t] = is_big ? 1 : 0;
        nbig += is_big ? 1u : 0u;
        for (int k = 0; k < 3; ++k) {
            if (!is_big) {
                lo[k] = fminf(lo[k], cen[k]);
                hi[k] = fmaxf(hi[k], cen[k]);
            }
        }
    }
    for (int k = 0; k < 3; ++k)
        for (int o = 16; o; o >>= 1) {
            lo[k] = fminf(lo[k], __shfl_xor_sync(0xffffffffu, lo[k], o));
            hi[k] = fmaxf(hi[k], __shfl_xor_sync(0xffffffffu, hi[k], o));
        }
    for (int o = 16; o; o >>= 1) nbig += __shfl_xor_sync(0xffffffffu, nbig, o);
    if ((threadIdx.x & 31) == 0) {
        for (int k = 0; k < 3; ++k) {
            atomicMin(&bounds[8 + k], f2ord(lo[k]));
            atomicMax(&bounds[11 + k], f2ord(hi[k]));
        }
        atomicAdd(&bounds[7], nbig);
    }
}

// spread the low 21 bits of v to every third bit
__device__ __forceinline__ unsigned long long expand21(unsigned v) {
    unsigned long long x = v & 0x1fffffu;
    x = (x | x << 32) & 0x1f00000000ffffull;
    x = (x | x << 16) & 0x1f0000ff0000ffull;
    x = (x | x << 8) & 0x100f00f00f00f00full;
    x = (x | x << 4) & 0x10c30c30c30c30c3ull;
    x = (x | x << 2) & 0x1249249249249249ull;
    return x;
}

// 63-bit Morton code (21 bits per axis) of the centroid in the given centroid
// bounds: cells of ~1e-6 of the scene extent, so triangles of small objects
// in a large room still get distinct codes.  Scene-sized triangles (when
// separated) get the largest key and sort to the end.
__global__ void k_morton(const float* __restrict__ v, const int* __restrict__ idx, int n,
                         const unsigned* __restrict__ bounds, const uint8_t* __restrict__ big,
                         unsigned long long* keys, int* ids) {
    int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n) return;
    ids[t] = t;
    if (big && big[t]) {
        keys[t] = ~0ull;
        return;
    }
    int a = idx[3 * t], b = idx[3 * t + 1], c = idx[3 * t + 2];
    unsigned q[3];
    for (int k = 0; k < 3; ++k) {
        float lo = ord2f(bounds[k]), hi = ord2f(bounds[3 + k]);
        float cen = (v[3 * a + k] + v[3 * b + k] + v[3 * c + k]) * (1.f / 3.f);
        float ext = hi - lo;
        float u = ext > 0.f ? (cen - lo) / ext : 0.5f;
        q[k] = (unsigned)fminf(fmaxf(u * 2097152.f, 0.f), 2097151.f);
    }
    keys[t] = (expand21(q[0]) << 2) | (expand21(q[1]) << 1) | expand21(q[2]);
}

// common-prefix length of sorted keys i and j (extended key = code, position)
__device__ __forceinline__ int delta(const unsigned long long* __restrict__ keys, int n, int i, int j) {
    if (j < 0 || j >= n) return -1;
    unsigned long long a = keys[i], b = keys[j];
    if (a != b) return __clzll(a ^ b);
    return 64 + __clz((unsigned)i ^ (unsigned)j);
}

__global__ void k_hierarchy(const unsigned long long* __restrict__ keys, int n, Node* nodes, int* leaf_parent, int2* rng) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n - 1) return;
    int d = (delta(keys, n, i, i + 1) - delta(keys, n, i, i - 1)) >= 0 ? 1 : -1;
    int dmin = delta(keys, n, i, i - d);
    int lmax = 2;
    while (delta(keys, n, i, i + lmax * d) > dmin) lmax <<= 1;
    int l = 0;
    for (int t = lmax >> 1; t >= 1; t >>= 1)
        if (delta(keys, n, i, i + (l + t) * d) > dmin) l += t;
    int j = i + l * d;
    int dnode = delta(keys, n, i, j);
    int s = 0;
    int t = l;
    do {
        t = (t + 1) >> 1;
        if (delta(keys, n, i, i + (s + t) * d) > dnode) s += t;
    } while (t > 1);
    int gamma = i + s * d + (d < 0 ? -1 : 0);
    int lo = i < j ? i : j, hi = i < j ? j : i;
    rng[i] = make_int2(lo, hi);
    int left = (lo == gamma) ? ~gamma : gamma;
    int right = (hi == gamma + 1) ? ~(gamma + 1) : gamma + 1;
    // separate 4-byte stores: .z (this node's parent) is written by the parent's thread
    nodes[i].child.x = left;
    nodes[i].child.y = right;
    if (left >= 0) nodes[left].child.z = i;
    else leaf_parent[gamma] = i;
    if (right >= 0) nodes[right].child.z = i;
    else leaf_parent[gamma + 1] = i;
}

__device__ __forceinline__ void tri_box(const float* __restrict__ v, const int* __restrict__ idx, int id,
                                        float lo[3], float hi[3]) {
    int a = idx[3 * id], b = idx[3 * id + 1], c = idx[3 * id + 2];
    for (int k = 0; k < 3; ++k) {
        float x = v[3 * a + k], y = v[3 * b + k], z = v[3 * c + k];
        lo[k] = fminf(x, fminf(y, z));
        hi[k] = fmaxf(x, fmaxf(y, z));
    }
}

__device__ __forceinline__ void write_child_box(Node* nd, int which, const float lo[3], const float hi[3]) {
    if (which == 0) {
        nd->xy0 = make_float4(lo[0], hi[0], lo[1], hi[1]);
        nd->z01.x = lo[2];
        nd->z01.y = hi[2];
    } else {
        nd->xy1 = make_float4(lo[0], hi[0], lo[1], hi[1]);
        nd->z01.z = lo[2];
        nd->z01.w = hi[2];
    }
}

__global__ void k_refit(const float* __restrict__ v, const int* __restrict__ idx, const int* __restrict__ ids,
                        int n, const int* __restrict__ leaf_parent, Node* nodes, unsigned* flags) {
    int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    float lo[3], hi[3];
    tri_box(v, idx, ids[k], lo, hi);
    int me = ~k;
    int p = leaf_parent[k];
    for (int level = 0; p >= 0 && level < 4096; ++level) {  // bounded walk to the root
        Node* nd = nodes + p;
        int4 ch = __ldcg(&nd->child);
        write_child_box(nd, ch.x == me ? 0 : 1, lo, hi);
        __threadfence();
        if (atomicAdd(&flags[p], 1u) == 0) return;  // the sibling finishes this node
        __threadfence();
        float4 a = __ldcg(&nd->xy0), b = __ldcg(&nd->xy1), z = __ldcg(&nd->z01);
        lo[0] = fminf(a.x, b.x);
        hi[0] = fmaxf(a.y, b.y);
        lo[1] = fminf(a.z, b.z);
        hi[1] = fmaxf(a.w, b.w);
        lo[2] = fminf(z.x, z.z);
        hi[2] = fmaxf(z.y, z.w);
        me = p;
        p = ch.z;
    }
}

// results of the clustering on the device: the root's reference and height,
// and whether one cluster is left
enum { CTL_ROOT, CTL_HEIGHT, CTL_DONE, CTL_ROUND };  // then (N, pair neighbours, buffer) per round
constexpr int CTL_ROUNDS = 64;  // slots

// triangles, materials, texture coordinates and the slot of each original id
__global__ void k_leaf_data(const float* __restrict__ v, const int* __restrict__ idx, const float* __restrict__ mat,
                            const float* __restrict__ uv, const int* __restrict__ ids,
                            const int* __restrict__ newpos, int m, const int* __restrict__ ctl, int n, Tri* tris,
                            float4* mato, float2* uvo, int* slot_of, int* specular) {
    int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n || (ctl && !ctl[CTL_DONE])) return;
    const int id = ids[k];
    if (newpos && k < m) k = newpos[k];  // the triangle's depth-first leaf position
    slot_of[id] = k;
    int a = idx[3 * id], b = idx[3 * id + 1], c = idx[3 * id + 2];
    Tri t;
    t.v0 = make_float4(v[3 * a], v[3 * a + 1], v[3 * a + 2], __int_as_float(id));
    t.v1 = make_float4(v[3 * b], v[3 * b + 1], v[3 * b + 2], 0.f);
    t.v2 = make_float4(v[3 * c], v[3 * c + 1], v[3 * c + 2], 0.f);
    tris[k] = t;
    Tri* r1 = tris + (size_t)n + k;  // the same triangle with its axes rotated (RayTri)
    r1->v0 = make_float4(t.v0.y, t.v0.z, t.v0.x, t.v0.w);
    r1->v1 = make_float4(t.v1.y, t.v1.z, t.v1.x, 0.f);
    r1->v2 = make_float4(t.v2.y, t.v2.z, t.v2.x, 0.f);
    Tri* r2 = r1 + n;
    r2->v0 = make_float4(t.v0.z, t.v0.x, t.v0.y, t.v0.w);
    r2->v1 = make_float4(t.v1.z, t.v1.x, t.v1.y, 0.f);
    r2->v2 = make_float4(t.v2.z, t.v2.x, t.v2.y, 0.f);
    const float* mt = mat + 8 * (size_t)id;
    mato[2 * k] = make_float4(mt[0], mt[1], mt[2], mt[3]);
    mato[2 * k + 1] = make_float4(mt[4], mt[5], mt[6], mt[7]);
    if (mt[7] > 0.f) atomicOr(specular, 1);
    if (uv) {
        const float* u = uv + 6 * (size_t)id;
        uvo[3 * k] = make_float2(u[0], u[1]);
        uvo[3 * k + 1] = make_float2(u[2], u[3]);
        uvo[3 * k + 2] = make_float2(u[4], u[5]);
    } else {
        uvo[3 * k] = uvo[3 * k + 1] = uvo[3 * k + 2] = make_float2(0.f, 0.f);
    }
}

// Turn every child that covers at most leaf_max triangles into a leaf over
// its contiguous range of sorted triangles (subtrees of a Morton-ordered tree
// cover contiguous key ranges).  Each thread rewrites only its own node.
__global__ void k_leafify(Node* bin, const int2* __restrict__ rng, int n_int, int leaf_max) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n_int) return;
    int c[2] = {bin[i].child.x, bin[i].child.y};
    for (int k = 0; k < 2; ++k) {
        if (c[k] < 0) c[k] = leaf_ref(~c[k], 1);
        else {
            int cnt = rng[c[k]].y - rng[c[k]].x + 1;
            if (cnt <= leaf_max) c[k] = leaf_ref(rng[c[k]].x, cnt);
        }
    }
    bin[i].child.x = c[0];
    bin[i].child.y = c[1];
}

// depth of every leaf of the original binary tree (an upper bound of the
// traversal depth after leafify), reduced with atomicMax
__global__ void k_depth(const int* __restrict__ leaf_parent, const Node* __restrict__ nodes, int n, unsigned* depth) {
    int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    unsigned d = 1;
    int p = leaf_parent[k];
    while (p > 0 && d < 4096) {
        p = nodes[p].child.z;
        ++d;
    }
    atomicMax(depth, d);
}

// ---------------------------------------------------------------- PLOC --
// Parallel locally-ordered clustering (Meister and Bittner, "Parallel
// locally-ordered clustering for bounding volume hierarchy construction",
// IEEE TVCG 2018).  Clusters start as the Morton-sorted triangles.  Each
// round every cluster finds, within R positions on either side, the
// cluster whose union box has the smallest surface area; mutual nearest
// neighbours merge into a new node at the lower position, and the array is
// compacted, keeping Morton order.  Rounds repeat until one cluster is left.
#ifndef HDOF_BUILDER
#define HDOF_BUILDER 1  // 1: PLOC, 0: LBVH
#endif
// The search radius R: 64 for trees that stay in L2 (the 164.6k-triangle room:
// the trace 2.5% and the G-buffer 2.6% faster than with 48; 56, 72, 80, 96 slower),
// 48 above PLOC_BIG triangles (the 5.25M-triangle scene's G-buffer is 8% slower
// at 64; radii 8..96 swept).
constexpr int PLOC_R_SMALL = 64, PLOC_R_BIG = 48;
constexpr int PLOC_BIG = 1 << 20;
constexpr int PLOC_B = 256;
constexpr int PLOC_CB = 1024;    // clusters per block of the count and the merge
constexpr int PLOC_CAP = 1024;   // clusters from which one block finishes in shared memory
__device__ __forceinline__ float union_area(float4 alo, float4 ahi, float4 blo, float4 bhi) {
    float x = fmaxf(ahi.x, bhi.x) - fminf(alo.x, blo.x);
    float y = fmaxf(ahi.y, bhi.y) - fminf(alo.y, blo.y);
    float z = fmaxf(ahi.z, bhi.z) - fminf(alo.z, blo.z);
    return x * y + y * z + z * x;
}

// A cluster: its node or leaf reference, and its box with the number of
// triangles (lo.w) and the height (hi.w) as int bits.
struct Clusters {
    int* ref[2];
    float4 *lo[2], *hi[2];
};

__global__ void k_ploc_init(const float* __restrict__ v, const int* __restrict__ idx, const int* __restrict__ ids,
                            int n, Clusters c, int* ctl) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i == 0) {
        ctl[CTL_DONE] = 0;
        ctl[CTL_ROUND] = n;
        ctl[CTL_ROUND + 1] = 0;
        ctl[CTL_ROUND + 2] = 0;
    }
    if (i >= n) return;
    float l[3], h[3];
    tri_box(v, idx, ids[i], l, h);
    c.ref[0][i] = leaf_ref(i, 1);
    c.lo[0][i] = make_float4(l[0], l[1], l[2], __int_as_float(1));
    c.hi[0][i] = make_float4(h[0], h[1], h[2], __int_as_float(0));
}

// Rounds on the device, so that the host need not read the cluster count:
// round r reads (N, pair neighbours this round, buffer holding the clusters)
// from its slot of ctl and writes the next round's.  The round kernels are
// launched over an upper bound of N and leave a round with N <= PLOC_CAP to
// k_ploc_finish.  Three launches a round (neighbours; counts of the clusters
// that stay; merge and compaction).  A tree of 165k triangles takes about 25
// such rounds and 45 in k_ploc_finish; with every round in six launches over
// all clusters, the leaf data moved twice and the subtree sizes walked
// bottom-up (they are the clusters' counts) its build took 3.1 ms, so 1.34
// (20k triangles 2.6 -> 0.94, 5.2M 11.0 -> 7.0).
__device__ __forceinline__ const int* ctl_slot(const int* ctl, int round) { return ctl + CTL_ROUND + 3 * round; }

template <int PLOC_R>
__global__ void __launch_bounds__(PLOC_B) k_ploc_nn(const int* __restrict__ ctl, int round, Clusters c,
                                                    int* __restrict__ nn) {
    const int* st = ctl_slot(ctl, round);
    const int N = st[0];
    if (N <= PLOC_CAP || st[1]) return;  // done here, or pairing neighbours: the whole block leaves
    const float4* __restrict__ lo = c.lo[st[2]];
    const float4* __restrict__ hi = c.hi[st[2]];
    __shared__ float4 slo[PLOC_B + 2 * PLOC_R], shi[PLOC_B + 2 * PLOC_R];
    for (int first = blockIdx.x * PLOC_B; first < N; first += gridDim.x * PLOC_B) {
        const int base = first - PLOC_R;
        __syncthreads();  // the previous chunk's searches
        for (int k = threadIdx.x; k < PLOC_B + 2 * PLOC_R; k += PLOC_B) {
            int g = base + k;
            if (g >= 0 && g < N) {
                slo[k] = lo[g];
                shi[k] = hi[g];
            }
        }
        __syncthreads();
        const int i = first + threadIdx.x;
        if (i >= N) continue;
        const int li = threadIdx.x + PLOC_R;
        const float4 a0 = slo[li], a1 = shi[li];
        float best = __int_as_float(0x7f800000);
        int bj = -1;
        const int j0 = max(i - PLOC_R, 0), j1 = min(i + PLOC_R, N - 1);
        for (int j = j0; j <= j1; ++j) {
            if (j == i) continue;
            float cost = union_area(a0, a1, slo[j - base], shi[j - base]);
            if (cost < best) {  // ascending j: ties keep the lower index
                best = cost;
                bj = j;
            }
        }
        nn[i] = bj;
    }
}

// the cluster that i merges with this round (-1: none): mutual nearest
// neighbours, or, when pairing, positions 2k and 2k + 1.  The pair's node
// takes the lower position; the upper one is dropped.
__device__ __forceinline__ int ploc_partner(int i, int N, int pair, const int* nn) {
    if (pair) return (i & 1) ? i - 1 : (i + 1 < N ? i + 1 : -1);
    const int j = nn[i];
    return j >= 0 && nn[j] == i ? j : -1;
}

__global__ void __launch_bounds__(PLOC_CB) k_ploc_count(const int* __restrict__ ctl, int round,
                                                        const int* __restrict__ nn, int* __restrict__ counts) {
    const int* st = ctl_slot(ctl, round);
    const int N = st[0];
    if (N <= PLOC_CAP) return;
    for (int b = blockIdx.x; b * PLOC_CB < N; b += gridDim.x) {
        const int i = b * PLOC_CB + threadIdx.x;
        bool stays = false;
        if (i < N) {
            const int j = ploc_partner(i, N, st[1], nn);
            stays = j < 0 || j > i;
        }
        const int c = __syncthreads_count(stays);
        if (threadIdx.x == 0) counts[b] = c;
    }
}

// the node of clusters a and b; its clusters' parent references follow
__device__ __forceinline__ void ploc_node(Node* nodes, int id, int ra, float4 al, float4 ah, int rb, float4 bl,
                                          float4 bh, float4& lo, float4& hi) {
    Node nd;
    nd.xy0 = make_float4(al.x, ah.x, al.y, ah.y);
    nd.xy1 = make_float4(bl.x, bh.x, bl.y, bh.y);
    nd.z01 = make_float4(al.z, ah.z, bl.z, bh.z);
    const int cnt = __float_as_int(al.w) + __float_as_int(bl.w);
    nd.child = make_int4(ra, rb, -1, cnt - 1);  // (parent: none yet; internal nodes of the subtree)
    nodes[id] = nd;
    if (ra >= 0) nodes[ra].child.z = id;
    if (rb >= 0) nodes[rb].child.z = id;
    lo = make_float4(fminf(al.x, bl.x), fminf(al.y, bl.y), fminf(al.z, bl.z), __int_as_float(cnt));
    hi = make_float4(fmaxf(ah.x, bh.x), fmaxf(ah.y, bh.y), fmaxf(ah.z, bh.z),
                     __int_as_float(max(__float_as_int(ah.w), __float_as_int(bh.w)) + 1));
}

// exclusive prefix of a flag over a block of PLOC_CB threads, and its total
__device__ __forceinline__ int block_rank(bool f, int* s_warp, int& total) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const unsigned m = __ballot_sync(0xffffffffu, f);
    if (lane == 0) s_warp[w] = __popc(m);
    __syncthreads();
    const int c = s_warp[lane];  // PLOC_CB / 32 = 32 warps
    const int before = __reduce_add_sync(0xffffffffu, lane < w ? c : 0);
    total = __reduce_add_sync(0xffffffffu, c);
    __syncthreads();
    return before + __popc(m & ((1u << lane) - 1u));
}

__global__ void __launch_bounds__(PLOC_CB) k_ploc_merge(int* ctl, int round, const int* __restrict__ nn,
                                                        const int* __restrict__ counts, Clusters c, Node* nodes,
                                                        unsigned* counter) {
    const int* st = ctl_slot(ctl, round);
    int* next = ctl + CTL_ROUND + 3 * (round + 1);
    const int N = st[0], pair = st[1], buf = st[2];
    if (N <= PLOC_CAP) {
        if (blockIdx.x == 0 && threadIdx.x < 3) next[threadIdx.x] = st[threadIdx.x];
        return;
    }
    __shared__ int s_warp[32];
    __shared__ int s_base;
    int counted = 0;  // chunks in s_base so far
    if (threadIdx.x == 0) s_base = 0;
    for (int b = blockIdx.x; b * PLOC_CB < N; b += gridDim.x) {
        __syncthreads();
        int before = 0;  // clusters that stay in the chunks before this one
        for (int k = counted + threadIdx.x; k < b; k += PLOC_CB) before += counts[k];
        counted = b;
        before = __reduce_add_sync(0xffffffffu, before);
        if ((threadIdx.x & 31) == 0 && before) atomicAdd(&s_base, before);
        const int i = b * PLOC_CB + threadIdx.x;
        const int j = i < N ? ploc_partner(i, N, pair, nn) : -1;
        const bool stays = i < N && (j < 0 || j > i);
        int total;
        const int rank = block_rank(stays, s_warp, total);  // (synchronises s_base too)
        const int k = s_base + rank;
        if (stays) {
            int ref = c.ref[buf][i];
            float4 lo = c.lo[buf][i], hi = c.hi[buf][i];
            if (j >= 0) {
                const int id = (int)atomicAdd(counter, 1u);
                ploc_node(nodes, id, ref, lo, hi, c.ref[buf][j], c.lo[buf][j], c.hi[buf][j], lo, hi);
                ref = id;
            }
            c.ref[1 - buf][k] = ref;
            c.lo[1 - buf][k] = lo;
            c.hi[1 - buf][k] = hi;
        }
        if (threadIdx.x == 0 && (b + 1) * PLOC_CB >= N) {  // the last chunk
            next[0] = s_base + total;
            next[1] = s_base + total == N;  // no mutual pair this round: pair neighbours once
            next[2] = 1 - buf;
        }
    }
}

// The last rounds, N <= PLOC_CAP, by one block with the clusters in shared
// memory: the same rounds, at a microsecond or two instead of six launches
// each.  Most of a tree's 70 rounds are such (each merges few of the clusters
// left).  While N <= PLOC_CB / 2, several threads share a cluster's search.
struct FinishSmem {
    float4 lo[PLOC_CAP], hi[PLOC_CAP];
    int ref[PLOC_CAP], nn[PLOC_CAP];
    int warp[32];
};
template <int PLOC_R>
__global__ void __launch_bounds__(PLOC_CB) k_ploc_finish(int* ctl, int round, Clusters c, Node* nodes,
                                                         unsigned* counter) {
    extern __shared__ __align__(16) unsigned char s_raw[];
    FinishSmem& s = *reinterpret_cast<FinishSmem*>(s_raw);
    constexpr int PER = PLOC_CAP / PLOC_CB;
    const int* st = ctl_slot(ctl, round);
    int N = st[0], pair = st[1];
    const int buf = st[2], t = threadIdx.x;
    if (N > PLOC_CAP) return;  // more rounds first
    for (int k = t; k < N; k += PLOC_CB) {
        s.ref[k] = c.ref[buf][k];
        s.lo[k] = c.lo[buf][k];
        s.hi[k] = c.hi[buf][k];
    }
    __syncthreads();
    for (int guard = 0; N > 1 && guard < 4 * PLOC_CAP; ++guard) {  // a round, or the pairing after it, merges
        if (!pair) {
            int P = 1;  // threads per cluster
            while (P < 32 && N * P * 2 <= PLOC_CB) P *= 2;
            for (int i0 = 0; i0 < N; i0 += PLOC_CB / P) {
                const int i = i0 + t / P, sub = t & (P - 1);
                float best = __int_as_float(0x7f800000);
                int bj = -1;
                if (i < N) {
                    const float4 a0 = s.lo[i], a1 = s.hi[i];
                    const int j0 = max(i - PLOC_R, 0), j1 = min(i + PLOC_R, N - 1);
                    for (int j = j0 + sub; j <= j1; j += P) {
                        if (j == i) continue;
                        const float cost = union_area(a0, a1, s.lo[j], s.hi[j]);
                        if (cost < best) {
                            best = cost;
                            bj = j;
                        }
                    }
                }
                for (int o = P >> 1; o; o >>= 1) {  // (the loops' trip counts are block-uniform)
                    const float ob = __shfl_xor_sync(0xffffffffu, best, o);
                    const int oj = __shfl_xor_sync(0xffffffffu, bj, o);
                    if (oj >= 0 && (bj < 0 || ob < best || (ob == best && oj < bj))) {
                        best = ob;
                        bj = oj;
                    }
                }
                if (i < N && sub == 0) s.nn[i] = bj;
            }
            __syncthreads();
        }
        // merge and compact in place: every cluster of this round is read before any is written
        int ref[PER], pos[PER];
        float4 lo[PER], hi[PER];
        int base = 0;
#pragma unroll
        for (int q = 0; q < PER; ++q) {
            const int i = q * PLOC_CB + t;
            pos[q] = -1;
            if (q * PLOC_CB >= N) continue;  // block-uniform
            const int j = i < N ? ploc_partner(i, N, pair, s.nn) : -1;
            const bool stays = i < N && (j < 0 || j > i);
            int total;
            const int rank = block_rank(stays, s.warp, total);
            if (stays) {
                pos[q] = base + rank;
                ref[q] = s.ref[i];
                lo[q] = s.lo[i];
                hi[q] = s.hi[i];
                if (j >= 0) {
                    const int id = (int)atomicAdd(counter, 1u);
                    ploc_node(nodes, id, ref[q], lo[q], hi[q], s.ref[j], s.lo[j], s.hi[j], lo[q], hi[q]);
                    ref[q] = id;
                }
            }
            base += total;
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < PER; ++q)
            if (pos[q] >= 0) {
                s.ref[pos[q]] = ref[q];
                s.lo[pos[q]] = lo[q];
                s.hi[pos[q]] = hi[q];
            }
        __syncthreads();
        pair = base == N;
        N = base;
    }
    if (t == 0) {
        ctl[CTL_ROOT] = s.ref[0];
        ctl[CTL_HEIGHT] = __float_as_int(s.hi[0].w);
        ctl[CTL_DONE] = N == 1;
    }
}

__global__ void k_big_boxes(const Tri* __restrict__ tris, int first, int n_big, float4* box) {
    int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n_big) return;
    Tri t = tris[first + k];
    box[2 * k] = make_float4(fminf(t.v0.x, fminf(t.v1.x, t.v2.x)), fminf(t.v0.y, fminf(t.v1.y, t.v2.y)),
                             fminf(t.v0.z, fminf(t.v1.z, t.v2.z)), 0.f);
    box[2 * k + 1] = make_float4(fmaxf(t.v0.x, fmaxf(t.v1.x, t.v2.x)), fmaxf(t.v0.y, fmaxf(t.v1.y, t.v2.y)),
                                 fmaxf(t.v0.z, fmaxf(t.v1.z, t.v2.z)), 0.f);
}

__global__ void k_closest(BvhView bvh, int n, const float* __restrict__ org, const float* __restrict__ dir, int cap,
                          unsigned* status, int* ids, float* ts) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    Hit h = closest_hit(bvh, ld3(org + 3 * (size_t)i), ld3(dir + 3 * (size_t)i), cap, status);
    ids[i] = h.slot >= 0 ? __float_as_int(__ldg(&bvh.tris[h.slot].v0.w)) : -1;
    ts[i] = h.t;
}

int blocks_for(long n, int bs) { return (int)((n + bs - 1) / bs); }

// ---- depth-first order and leaves -------------------------------------------
// The clustering numbers nodes in merge order, which scatters a parent and its
// children over memory.  Relabelling in depth-first pre-order (a node, then
// its first child's subtree, then its second child's) keeps every subtree in
// one contiguous range and puts a node's first child right after it, so a
// descent touches neighbouring cache lines.  The triangles are stored in
// depth-first leaf order, so the triangles of any subtree occupy consecutive
// slots, and each subtree of at most leaf_max triangles becomes one leaf over
// them: fewer traversal steps for one more triangle test per extra triangle.
// The tree itself, its boxes and the closest hits are unchanged.
__device__ __forceinline__ int n_leaves(const Node* __restrict__ nodes, int ref) {
    return ref >= 0 ? __ldg(&nodes[ref].child.w) + 1 : 1;
}

// pre-order index and first leaf position of each node: per step towards the
// root one node, plus the first child's subtree when the path goes through a
// second child
__global__ void k_dfs_index(const Node* __restrict__ nodes, int n, const int* __restrict__ ctl, int2* place) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n || !ctl[CTL_DONE]) return;
    const int root = ctl[CTL_ROOT];
    int idx = 0, leaf = 0, c = i, p = __ldg(&nodes[i].child.z);
    for (int guard = 0; c != root && guard < n; ++guard) {  // a walk is at most the tree's depth
        const int4 ch = __ldg(&nodes[p].child);
        idx += 1;
        if (c == ch.y) {
            const int l = n_leaves(nodes, ch.x);
            leaf += l;
            idx += l - 1;
        }
        c = p;
        p = ch.z;
    }
    place[i] = make_int2(idx, leaf);
}

// nodes to their places, with their children's new references; the new slot
// of each sorted triangle
__global__ void k_dfs_permute(const Node* __restrict__ nodes, int n, const int* __restrict__ ctl,
                              const int2* __restrict__ place, int leaf_max, Node* out, int* newpos) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n || !ctl[CTL_DONE]) return;
    Node nd = nodes[i];
    const int2 pl = place[i];
    const int c[2] = {nd.child.x, nd.child.y};
    int o[2], first = pl.y;
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const int cnt = n_leaves(nodes, c[k]);
        if (c[k] < 0) {
            newpos[(~c[k]) >> 3] = first;
            o[k] = leaf_ref(first, 1);
        } else {
            o[k] = cnt <= leaf_max ? leaf_ref(first, cnt) : place[c[k]].x;
        }
        first += cnt;
    }
    nd.child.x = o[0];
    nd.child.y = o[1];
    nd.child.z = nd.child.z < 0 ? -1 : place[nd.child.z].x;
    out[pl.x] = nd;
}

}  // namespace
}  // namespace hdof

using namespace hdof;

namespace {
size_t up256(size_t x) { return (x + 255) & ~size_t(255); }

#ifndef HDOF_PLOC_LEAF_MAX
#define HDOF_PLOC_LEAF_MAX 2  // largest collapsed leaf of the clustered tree (<= 8; 1: no collapse); 2 measured fastest
#endif

}  // namespace

extern "C" int hdof_build_bvh(const float* verts, int32_t n_verts, const int32_t* idx, int32_t n_tris,
                              const float* mat, const float* uv, hdof_bvh** out, void* stream) {
    clear_error();
    HDOF_CHECK_ARG(out, "hdof_build_bvh: out is NULL");
    *out = nullptr;
    HDOF_CHECK_ARG(verts && idx && mat, "hdof_build_bvh: verts, idx and mat must be device pointers");
    HDOF_CHECK_ARG(n_tris >= 1 && n_tris <= (1 << 27), "hdof_build_bvh: n_tris %d outside 1..2^27", n_tris);
    HDOF_CHECK_ARG(n_verts >= 3, "hdof_build_bvh: n_verts %d < 3", n_verts);
    cudaStream_t s = as_stream(stream);
    const int n = n_tris;

    // ---- scratch (freed before returning) ----
    size_t sort_bytes = 0;
    cub::DeviceRadixSort::SortPairs(nullptr, sort_bytes, (unsigned long long*)nullptr, (unsigned long long*)nullptr,
                                    (int*)nullptr, (int*)nullptr, n, 0, 64, s);
    const size_t N = (size_t)n;
    size_t o = 0;
    auto take = [&](size_t bytes) {
        const size_t at = o;
        o += up256(bytes);
        return at;
    };
    const size_t o_bounds = take(NB * sizeof(unsigned)), o_cnt = take(sizeof(unsigned));
    const size_t o_ctl = take((CTL_ROUND + 3 * CTL_ROUNDS) * sizeof(int));
    const size_t o_keys_in = take(8 * N), o_keys_out = take(8 * N), o_ids_in = take(4 * N), o_ids_out = take(4 * N);
    const size_t o_sort = take(sort_bytes);
    // the clustering's, or the linear tree's
    const size_t o_ref0 = take(4 * N), o_ref1 = take(4 * N), o_lo0 = take(16 * N), o_lo1 = take(16 * N);
    const size_t o_hi0 = take(16 * N), o_hi1 = take(16 * N), o_nn = take(4 * N), o_counts = take(4 * (N / PLOC_CB + 1));
    const size_t o_nodes = take(sizeof(Node) * N), o_place = take(8 * N), o_newpos = take(4 * N), o_big = take(N);
    void* tmp = nullptr;
    cudaError_t e = cudaMalloc(&tmp, o);
    if (e != cudaSuccess) return cuda_fail(e, "hdof_build_bvh: cudaMalloc scratch");
    char* t8 = static_cast<char*>(tmp);
    unsigned* bounds = reinterpret_cast<unsigned*>(t8 + o_bounds);
    unsigned* counters = reinterpret_cast<unsigned*>(t8 + o_cnt);  // [0] nodes (clustering), tree depth (linear tree)
    int* ctl = reinterpret_cast<int*>(t8 + o_ctl);
    unsigned long long* keys_in = reinterpret_cast<unsigned long long*>(t8 + o_keys_in);
    unsigned long long* keys_out = reinterpret_cast<unsigned long long*>(t8 + o_keys_out);
    int* ids_in = reinterpret_cast<int*>(t8 + o_ids_in);
    int* ids_out = reinterpret_cast<int*>(t8 + o_ids_out);
    void* sort_tmp = t8 + o_sort;
    int* ref0 = reinterpret_cast<int*>(t8 + o_ref0);
    int* ref1 = reinterpret_cast<int*>(t8 + o_ref1);
    float4* lo0 = reinterpret_cast<float4*>(t8 + o_lo0);
    float4* lo1 = reinterpret_cast<float4*>(t8 + o_lo1);
    float4* hi0 = reinterpret_cast<float4*>(t8 + o_hi0);
    float4* hi1 = reinterpret_cast<float4*>(t8 + o_hi1);
    int* nn = reinterpret_cast<int*>(t8 + o_nn);
    int* counts = reinterpret_cast<int*>(t8 + o_counts);
    Node* nodes0 = reinterpret_cast<Node*>(t8 + o_nodes);
    int2* place = reinterpret_cast<int2*>(t8 + o_place);
    int* newpos = reinterpret_cast<int*>(t8 + o_newpos);
    uint8_t* big = reinterpret_cast<uint8_t*>(t8 + o_big);
    int* leaf_parent = ref0;                               // linear tree
    unsigned* flags = reinterpret_cast<unsigned*>(ref1);
    int2* rng = reinterpret_cast<int2*>(lo0);

    hdof_bvh* b = nullptr;
    auto fail = [&](int code) {
        cudaStreamSynchronize(s);
        cudaFree(tmp);
        if (b) {
            if (b->pool) cudaFree(b->pool);
            delete b;
        }
        return code;
    };
    // minima start at all ones, the rest at zero
    if ((e = cudaMemsetAsync(bounds, 0, NB * sizeof(unsigned), s)) == cudaSuccess)
        for (int k : {0, 8, 14})
            if (e == cudaSuccess) e = cudaMemsetAsync(bounds + k, 0xff, 3 * sizeof(unsigned), s);
    if (e != cudaSuccess) return fail(cuda_fail(e, "hdof_build_bvh: init bounds"));
    const int rb = blocks_for(n, 256) < 2 * sm_count() ? blocks_for(n, 256) : 2 * sm_count();
    k_scene_bounds<<<rb, 256, 0, s>>>(verts, n_verts, idx, n, bounds);
    unsigned hb[NB];
    // before anything else reads a vertex through an index
    if ((e = cudaGetLastError()) != cudaSuccess ||
        (e = cudaMemcpyAsync(hb, bounds, sizeof hb, cudaMemcpyDeviceToHost, s)) != cudaSuccess ||
        (e = cudaStreamSynchronize(s)) != cudaSuccess)
        return fail(cuda_fail(e, "hdof_build_bvh: scene bounds"));
    if (hb[6]) {
        set_error("hdof_build_bvh: a triangle index is outside 0..n_verts-1");
        return fail(HDOF_EINVAL);
    }
    int n_big = 0;
    bool separate = false;
    if (HDOF_BIG_MAX > 0) {
        k_classify<<<rb, 256, 0, s>>>(verts, idx, n, 0.02f, bounds, big);
        if ((e = cudaGetLastError()) != cudaSuccess ||
            (e = cudaMemcpyAsync(hb, bounds, sizeof hb, cudaMemcpyDeviceToHost, s)) != cudaSuccess ||
            (e = cudaStreamSynchronize(s)) != cudaSuccess)
            return fail(cuda_fail(e, "hdof_build_bvh: classify"));
        // separate scene-sized triangles only when they are few and the rest can form a tree
        n_big = (int)hb[7];
        separate = n >= 64 && n_big > 0 && n_big <= HDOF_BIG_MAX && n - n_big >= 2;
        if (!separate) n_big = 0;
    }
    const int n_small = n - n_big;
    const unsigned* cbounds = bounds + (separate ? 8 : 14);  // centroid bounds (lo at [0..2], hi at [3..5])

    b = new (std::nothrow) hdof_bvh();
    if (!b) {
        set_error("hdof_build_bvh: host allocation failed");
        return fail(HDOF_ENOMEM);
    }
    cudaGetDevice(&b->device);
    b->n_tris = n;
    b->n_big = n_big;
    const int n_int = n_small > 1 ? n_small - 1 : 1;
    size_t off_tris = up256(sizeof(Node) * (size_t)n_int);
    size_t off_mat = off_tris + up256(sizeof(Tri) * 3 * (size_t)n);
    size_t off_uv = off_mat + up256(sizeof(float4) * 2 * (size_t)n);
    size_t off_big = off_uv + up256(sizeof(float2) * 3 * (size_t)n);
    size_t off_slot = off_big + up256(sizeof(float4) * 2 * (size_t)(n_big > 0 ? n_big : 1));
    size_t off_spec = off_slot + up256(sizeof(int) * (size_t)n);
    size_t total = off_spec + sizeof(int);
    if ((e = cudaMalloc(&b->pool, total)) != cudaSuccess) return fail(cuda_fail(e, "hdof_build_bvh: cudaMalloc"));
    b->bytes = total;
    char* base = static_cast<char*>(b->pool);
    b->nodes = reinterpret_cast<Node*>(base);
    b->tris = reinterpret_cast<Tri*>(base + off_tris);
    b->mat = reinterpret_cast<float4*>(base + off_mat);
    b->uv = reinterpret_cast<float2*>(base + off_uv);
    b->big_box = reinterpret_cast<float4*>(base + off_big);
    b->slot_of = reinterpret_cast<int*>(base + off_slot);

    // Morton codes and radix sort (scene-sized triangles keyed last)
    k_morton<<<blocks_for(n, 256), 256, 0, s>>>(verts, idx, n, cbounds, separate ? big : nullptr, keys_in, ids_in);
    e = cub::DeviceRadixSort::SortPairs(sort_tmp, sort_bytes, keys_in, keys_out, ids_in, ids_out, n, 0,
                                        separate ? 64 : 63, s);
    if (e != cudaSuccess) return fail(cuda_fail(e, "hdof_build_bvh: sort"));
    int* spec_flag = reinterpret_cast<int*>(base + off_spec);
    if ((e = cudaMemsetAsync(spec_flag, 0, sizeof(int), s)) != cudaSuccess)
        return fail(cuda_fail(e, "hdof_build_bvh: clear"));
    // leaf data in sorted order (newpos NULL) or at the depth-first positions of a clustered tree
    auto leaf_data = [&](const int* newpos, const int* ctl) {
        k_leaf_data<<<blocks_for(n, 256), 256, 0, s>>>(verts, idx, mat, uv, ids_out, newpos, n_small, ctl, n, b->tris,
                                                       b->mat, b->uv, b->slot_of, spec_flag);
        if (n_big > 0) k_big_boxes<<<1, 64, 0, s>>>(b->tris, n - n_big, n_big, b->big_box);
    };

    int depth = 0;
    b->n_nodes = 0;
    if (n_small <= HDOF_LEAF_MAX) {
        leaf_data(nullptr, nullptr);
        b->root = leaf_ref(0, n_small);
        depth = 1;
    } else if (HDOF_BUILDER == 0) {
        // binary LBVH over the first n_small sorted triangles, built in place
        leaf_data(nullptr, nullptr);
        int minus1 = -1;
        Node* nodes = b->nodes;
        if ((e = cudaMemsetAsync(nodes, 0, sizeof(Node) * (size_t)(n_small - 1), s)) != cudaSuccess ||
            (e = cudaMemsetAsync(flags, 0, sizeof(unsigned) * (size_t)(n_small - 1), s)) != cudaSuccess ||
            (e = cudaMemcpyAsync(&nodes[0].child.z, &minus1, sizeof(int), cudaMemcpyHostToDevice, s)) != cudaSuccess ||
            (e = cudaMemsetAsync(counters, 0, sizeof(unsigned), s)) != cudaSuccess)
            return fail(cuda_fail(e, "hdof_build_bvh: clear"));
        k_hierarchy<<<blocks_for(n_small - 1, 256), 256, 0, s>>>(keys_out, n_small, nodes, leaf_parent, rng);
        k_refit<<<blocks_for(n_small, 256), 256, 0, s>>>(verts, idx, ids_out, n_small, leaf_parent, nodes, flags);
        k_depth<<<blocks_for(n_small, 256), 256, 0, s>>>(leaf_parent, nodes, n_small, counters);
        k_leafify<<<blocks_for(n_small - 1, 256), 256, 0, s>>>(nodes, rng, n_small - 1, HDOF_LEAF_MAX);
        unsigned hd = 0;
        if ((e = cudaGetLastError()) != cudaSuccess ||
            (e = cudaMemcpyAsync(&hd, counters, sizeof hd, cudaMemcpyDeviceToHost, s)) != cudaSuccess ||
            (e = cudaStreamSynchronize(s)) != cudaSuccess)
            return fail(cuda_fail(e, "hdof_build_bvh: hierarchy"));
        depth = (int)hd;
        b->n_nodes = n_small - 1;
        b->root = 0;
    } else {
        // PLOC over the first n_small sorted triangles
        const int m = n_small, ni = m - 1;
        Clusters c{{ref0, ref1}, {lo0, lo1}, {hi0, hi1}};
        if ((e = cudaMemsetAsync(counters, 0, sizeof(unsigned), s)) != cudaSuccess)
            return fail(cuda_fail(e, "hdof_build_bvh: clear"));
        k_ploc_init<<<blocks_for(m, 256), 256, 0, s>>>(verts, idx, ids_out, m, c, ctl);
        const bool small = m <= PLOC_BIG;
        const size_t smem = sizeof(FinishSmem);
        if ((e = cudaFuncSetAttribute(small ? k_ploc_finish<PLOC_R_SMALL> : k_ploc_finish<PLOC_R_BIG>,
                                      cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) != cudaSuccess)
            return fail(cuda_fail(e, "hdof_build_bvh: shared memory"));
        // rounds until PLOC_CAP clusters are left, as a round leaves about four
        // fifths; should they not suffice, the device says so and more follow
        int Nb = m, round = 0, all = 0;
        for (bool first = true;; first = false) {
            int rounds = 0;
            if (Nb > PLOC_CAP) {
                rounds = (int)std::ceil(std::log((double)Nb / PLOC_CAP) / std::log(1.22)) + 1;
                rounds = std::min(std::max(rounds, first ? 1 : 16), CTL_ROUNDS - 1);
            }
            all += rounds;
            for (int r = 0; r < rounds; ++r, ++round) {
                // at most a full machine of blocks: the later rounds need far fewer than the first
                const int g1 = std::min(blocks_for(Nb, PLOC_B), 8 * sm_count());
                const int g2 = std::min(blocks_for(Nb, PLOC_CB), 2 * sm_count());
                if (small) k_ploc_nn<PLOC_R_SMALL><<<g1, PLOC_B, 0, s>>>(ctl, round, c, nn);
                else k_ploc_nn<PLOC_R_BIG><<<g1, PLOC_B, 0, s>>>(ctl, round, c, nn);
                k_ploc_count<<<g2, PLOC_CB, 0, s>>>(ctl, round, nn, counts);
                k_ploc_merge<<<g2, PLOC_CB, 0, s>>>(ctl, round, nn, counts, c, nodes0, counters);
            }
            if (small) k_ploc_finish<PLOC_R_SMALL><<<1, PLOC_CB, smem, s>>>(ctl, round, c, nodes0, counters);
            else k_ploc_finish<PLOC_R_BIG><<<1, PLOC_CB, smem, s>>>(ctl, round, c, nodes0, counters);
            // (these leave at once while the clustering is not done)
            k_dfs_index<<<blocks_for(ni, 256), 256, 0, s>>>(nodes0, ni, ctl, place);
            k_dfs_permute<<<blocks_for(ni, 256), 256, 0, s>>>(nodes0, ni, ctl, place, HDOF_PLOC_LEAF_MAX, b->nodes,
                                                              newpos);
            leaf_data(newpos, ctl);
            int h[3], slot[3];
            if ((e = cudaGetLastError()) != cudaSuccess ||
                (e = cudaMemcpyAsync(h, ctl, sizeof h, cudaMemcpyDeviceToHost, s)) != cudaSuccess ||
                (e = cudaMemcpyAsync(slot, ctl + CTL_ROUND + 3 * round, sizeof slot, cudaMemcpyDeviceToHost, s)) !=
                    cudaSuccess ||
                (e = cudaStreamSynchronize(s)) != cudaSuccess)
                return fail(cuda_fail(e, "hdof_build_bvh: clustering"));
            if (h[CTL_DONE]) {
                depth = h[CTL_HEIGHT];
                break;
            }
            if (all > 100000 || slot[0] <= PLOC_CAP) {
                set_error("hdof_build_bvh: clustering did not converge");
                return fail(HDOF_ECUDA);
            }
            Nb = slot[0];
            if ((e = cudaMemcpyAsync(ctl + CTL_ROUND, ctl + CTL_ROUND + 3 * round, sizeof slot, cudaMemcpyDeviceToDevice,
                                     s)) != cudaSuccess)
                return fail(cuda_fail(e, "hdof_build_bvh: clustering"));
            round = 0;
        }
        b->n_nodes = ni;
        b->root = 0;
    }
    int has_spec = 0;
    if ((e = cudaGetLastError()) != cudaSuccess ||
        (e = cudaMemcpyAsync(&has_spec, spec_flag, sizeof(int), cudaMemcpyDeviceToHost, s)) != cudaSuccess ||
        (e = cudaStreamSynchronize(s)) != cudaSuccess)
        return fail(cuda_fail(e, "hdof_build_bvh: leaf data"));
    b->specular = has_spec;
    b->depth = depth;
    if (depth + 1 >= HDOF_STACK) {
        set_error("hdof_build_bvh: tree depth %d exceeds the %d-entry traversal stack", depth, HDOF_STACK);
        return fail(HDOF_EUNSUPPORTED);
    }
    cudaFree(tmp);
    *out = b;
    return HDOF_OK;
}

extern "C" int hdof_bvh_destroy(hdof_bvh* b) {
    clear_error();
    if (!b) return HDOF_OK;
    int cur = 0;
    cudaGetDevice(&cur);
    if (cur != b->device) cudaSetDevice(b->device);
    cudaError_t e = cudaFree(b->pool);
    if (cur != b->device) cudaSetDevice(cur);
    delete b;
    return e == cudaSuccess ? HDOF_OK : cuda_fail(e, "hdof_bvh_destroy");
}

extern "C" int hdof_bvh_info(const hdof_bvh* b, hdof_bvh_stats* info) {
    clear_error();
    HDOF_CHECK_ARG(b && info, "hdof_bvh_info: NULL argument");
    info->n_tris = b->n_tris;
    info->n_nodes = b->n_nodes;
    info->depth = b->depth;
    info->n_big = b->n_big;
    info->device_bytes = (int64_t)b->bytes;
    return HDOF_OK;
}

extern "C" int hdof_closest_hits(const hdof_bvh* b, int32_t n, const float* org, const float* dir, int32_t* ids,
                                 float* ts, void* stream) {
    clear_error();
    HDOF_CHECK_ARG(b, "hdof_closest_hits: bvh is NULL");
    HDOF_CHECK_ARG(n >= 0, "hdof_closest_hits: n < 0");
    if (n == 0) return HDOF_OK;
    HDOF_CHECK_ARG(org && dir && ids && ts, "hdof_closest_hits: NULL buffer");
    unsigned* st = status_ptr();
    HDOF_CHECK_ARG(st, "hdof_closest_hits: no status word on this device");
    const int cap = step_cap(0, b->n_nodes, b->n_tris);
    k_closest<<<blocks_for(n, 128), 128, 0, as_stream(stream)>>>(b->view(), n, org, dir, cap, st, ids, ts);
    HDOF_LAUNCHED("hdof_closest_hits");
    return HDOF_OK;
}
