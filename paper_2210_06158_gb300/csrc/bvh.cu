// Device-built BVH of libdof (the acceleration structure whose build the paper
// counts in its ray-trace time, Section 4.2).
//
// Both builders start from the triangles sorted by the 63-bit Morton codes of their
// centroids (21 bits per axis: scenes with a ground plane hundreds of metres wide still
// resolve centimetre detail; a stable LSD radix sort written here, 8-bit digits,
// warp-matched ranks), the default one by as many of the upper bits as its triangles' size
// asks for (cluster_key_from).  The default one joins neighbours in one round of PLOC clustering
// and splits the clusters top-down by a binned surface-area heuristic.  The other is the
// LBVH after Karras, "Maximizing Parallelism in the Construction of BVHs, Octrees, and
// k-d Trees" (HPG 2012): one thread per internal node finds its key range and split
// (ties between equal codes broken by the sorted index), then a bottom-up box refit in
// which the second thread to reach a node merges its two children (atomic arrival
// counter, no waiting).  Nodes hold both child boxes so that traversal fetches one node
// per step.

#include "dof_internal.cuh"

#include <algorithm>
#include <cstring>

namespace {

__device__ __forceinline__ int ord_of(float f) {
    int i = __float_as_int(f);
    return i >= 0 ? i : i ^ 0x7FFFFFFF;
}
__device__ __forceinline__ float float_of(int i) { return __int_as_float(i >= 0 ? i : i ^ 0x7FFFFFFF); }

__device__ __forceinline__ float3 vtx(const float *xyz, uint32_t i) {
    return make_float3(xyz[3 * (size_t)i], xyz[3 * (size_t)i + 1], xyz[3 * (size_t)i + 2]);
}

// min (c < 3) and max (c >= 3) of v over the block, then one global atomic per component.
// The kernels that call it stride over their elements with a few blocks per SM: one set of
// atomics per warp of the whole input kept the six words' lines busy (64 us at 496k
// triangles; 8 us this way)
__device__ __forceinline__ void block_bounds(const float *v, int *out) {
    __shared__ int s[6];
    if (threadIdx.x < 6) s[threadIdx.x] = threadIdx.x < 3 ? 0x7FFFFFFF : (int)0x80000000;
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 6; k++) {
        const int o = ord_of(v[k]);
        const int w = k < 3 ? __reduce_min_sync(0xffffffffu, o) : __reduce_max_sync(0xffffffffu, o);
        if ((threadIdx.x & 31) == 0) {
            if (k < 3) atomicMin(&s[k], w);
            else atomicMax(&s[k], w);
        }
    }
    __syncthreads();
    if (threadIdx.x < 3) atomicMin(&out[threadIdx.x], s[threadIdx.x]);
    else if (threadIdx.x < 6) atomicMax(&out[threadIdx.x], s[threadIdx.x]);
}

// centroids and their bounds (order-preserving int atomics); flags bad indices
__global__ void __launch_bounds__(256) k_centroids(const float *xyz, uint32_t n_verts, const uint32_t *idx, uint32_t n,
                                                   float4 *cen, int *bounds, int *bad) {
    float v[6] = {INFINITY, INFINITY, INFINITY, -INFINITY, -INFINITY, -INFINITY};
    for (uint32_t t = blockIdx.x * blockDim.x + threadIdx.x; t < n; t += gridDim.x * blockDim.x) {
        uint32_t i0 = idx[3 * (size_t)t], i1 = idx[3 * (size_t)t + 1], i2 = idx[3 * (size_t)t + 2];
        if (i0 >= n_verts || i1 >= n_verts || i2 >= n_verts) {
            atomicExch(bad, 1);
            i0 = i1 = i2 = 0;
        }
        float3 a = vtx(xyz, i0), b = vtx(xyz, i1), d = vtx(xyz, i2);
        float3 lo = make_float3(fminf(a.x, fminf(b.x, d.x)), fminf(a.y, fminf(b.y, d.y)), fminf(a.z, fminf(b.z, d.z)));
        float3 hi = make_float3(fmaxf(a.x, fmaxf(b.x, d.x)), fmaxf(a.y, fmaxf(b.y, d.y)), fmaxf(a.z, fmaxf(b.z, d.z)));
        const float c[3] = {0.5f * (lo.x + hi.x), 0.5f * (lo.y + hi.y), 0.5f * (lo.z + hi.z)};
        cen[t] = make_float4(c[0], c[1], c[2], fmaxf(hi.x - lo.x, fmaxf(hi.y - lo.y, hi.z - lo.z)));
#pragma unroll
        for (int k = 0; k < 3; k++) { v[k] = fminf(v[k], c[k]); v[3 + k] = fmaxf(v[3 + k], c[k]); }
    }
    block_bounds(v, bounds);
}

// Threshold of a "large" triangle, kept out of the tree and tested by every ray: its largest
// box extent above `share` of the largest centroid extent of the scene.  The SAH splits take
// all but scene-spanning triangles (a ground plane) well, so only those above 1/2 stay out:
// every one costs every ray a test, and at 1/16 the small scene's 36 box faces did (a frame of
// 256 x 144 0.120 -> 0.117 ms, its tracer 0.047 -> 0.041 ms as packets).  The radix tree
// keeps 1/16: it splits by centroids alone, and one big box fattens every node above it.
constexpr float kLargeSah = 0.5f, kLargeLbvh = 1.f / 16.f;
__device__ __forceinline__ float big_threshold(const int *bounds, float share) {
    float e = 0.f;
    for (int k = 0; k < 3; k++) e = fmaxf(e, float_of(bounds[3 + k]) - float_of(bounds[k]));
    return e * share;
}

// count the large triangles and the centroid bounds of the others
__global__ void __launch_bounds__(256) k_classify(const float4 *cen, uint32_t n, const int *bounds, float share, int *n_big,
                                                  int *small_bounds) {
    const float thr = big_threshold(bounds, share);
    float v[6] = {INFINITY, INFINITY, INFINITY, -INFINITY, -INFINITY, -INFINITY};
    int nb = 0;
    for (uint32_t t = blockIdx.x * blockDim.x + threadIdx.x; t < n; t += gridDim.x * blockDim.x) {
        const float4 q = cen[t];
        if (q.w > thr) {
            nb++;
            continue;
        }
        const float c[3] = {q.x, q.y, q.z};
#pragma unroll
        for (int k = 0; k < 3; k++) { v[k] = fminf(v[k], c[k]); v[3 + k] = fmaxf(v[3 + k], c[k]); }
    }
    nb = __reduce_add_sync(0xffffffffu, nb);
    if ((threadIdx.x & 31) == 0 && nb) atomicAdd(n_big, nb);
    block_bounds(v, small_bounds);
}

// spread the low 21 bits of v to every third bit
__device__ __forceinline__ unsigned long long expand21(uint32_t v) {
    unsigned long long x = v & 0x1fffffull;
    x = (x | x << 32) & 0x1f00000000ffffull;
    x = (x | x << 16) & 0x1f0000ff0000ffull;
    x = (x | x << 8) & 0x100f00f00f00f00full;
    x = (x | x << 4) & 0x10c30c30c30c30c3ull;
    x = (x | x << 2) & 0x1249249249249249ull;
    return x;
}

// Morton keys over the centroid bounds `bounds`; with separate_big, large triangles
// (classified against `all_bounds`) get the key ~0 and sort after every other one
__global__ void k_morton(const float4 *cen, uint32_t n, const int *bounds, const int *all_bounds, float share, int separate_big,
                         unsigned long long *keys, uint32_t *vals) {
    uint32_t t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n) return;
    vals[t] = t;
    if (separate_big && cen[t].w > big_threshold(all_bounds, share)) {
        keys[t] = ~0ull;
        return;
    }
    float lo[3], ext[3];
    for (int k = 0; k < 3; k++) {
        lo[k] = float_of(bounds[k]);
        ext[k] = float_of(bounds[3 + k]) - lo[k];
    }
    float4 c = cen[t];
    float p[3] = {c.x, c.y, c.z};
    uint32_t q[3];
    for (int k = 0; k < 3; k++) {
        float u = ext[k] > 0.f ? (p[k] - lo[k]) / ext[k] : 0.f;
        q[k] = (uint32_t)fminf(fmaxf(u * 2097152.f, 0.f), 2097151.f);
    }
    keys[t] = (expand21(q[0]) << 2) | (expand21(q[1]) << 1) | expand21(q[2]);
}

// sorted triangles: v0 (w = original id), v1, v2 (w = material)
__global__ void k_sorted_tris(const float *xyz, const uint32_t *idx, const uint32_t *mat, uint32_t n,
                              uint32_t n_verts, const uint32_t *order, float4 *tris) {
    uint32_t k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    uint32_t t = order[k];
    uint32_t i0 = idx[3 * (size_t)t], i1 = idx[3 * (size_t)t + 1], i2 = idx[3 * (size_t)t + 2];
    if (i0 >= n_verts || i1 >= n_verts || i2 >= n_verts) i0 = i1 = i2 = 0;
    float3 a = vtx(xyz, i0), b = vtx(xyz, i1), c = vtx(xyz, i2);
    tris[3 * (size_t)k] = make_float4(a.x, a.y, a.z, __int_as_float((int)t));
    tris[3 * (size_t)k + 1] = make_float4(b.x, b.y, b.z, 0.f);
    tris[3 * (size_t)k + 2] = make_float4(c.x, c.y, c.z, __int_as_float(mat ? (int)mat[t] : 0));
}

// common-prefix length of sorted keys i and j, ties broken by index (Karras 2012)
__device__ __forceinline__ int delta(const unsigned long long *keys, int n, int i, int j) {
    if (j < 0 || j >= n) return -1;
    unsigned long long a = keys[i], b = keys[j];
    if (a != b) return __clzll((long long)(a ^ b));
    return 64 + __clz(i ^ j);
}

// one thread per internal node: its range, split and children; parent links.
// child refs: >= 0 internal, < 0 leaf ~k
__global__ void k_karras(const unsigned long long *keys, int n, int4 *child, int *parent_node, int *parent_leaf, int *bad) {
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
    int s = 0, t = l;
    do {
        t = (t + 1) >> 1;
        if (delta(keys, n, i, i + (s + t) * d) > dnode) s += t;
    } while (t > 1);
    int g = i + s * d + min(d, 0);
    int lo = min(i, j), hi = max(i, j);
    if (lo < 0 || hi > n - 1 || g < lo || g + 1 > hi) {   // cannot happen for a valid key order
        atomicExch(bad, 2);
        child[i] = make_int4(~0, ~0, 0, 0);
        return;
    }
    int left = (lo == g) ? ~g : g;
    int right = (hi == g + 1) ? ~(g + 1) : g + 1;
    child[i] = make_int4(left, right, 0, 0);
    if (left < 0) parent_leaf[~left] = i; else parent_node[left] = i;
    if (right < 0) parent_leaf[~right] = i; else parent_node[right] = i;
    if (i == 0) parent_node[0] = -1;
}

__device__ __forceinline__ void tri_box(const float4 *tris, int k, float3 &lo, float3 &hi) {
    float4 a = tris[3 * (size_t)k], b = tris[3 * (size_t)k + 1], c = tris[3 * (size_t)k + 2];
    lo = make_float3(fminf(a.x, fminf(b.x, c.x)), fminf(a.y, fminf(b.y, c.y)), fminf(a.z, fminf(b.z, c.z)));
    hi = make_float3(fmaxf(a.x, fmaxf(b.x, c.x)), fmaxf(a.y, fmaxf(b.y, c.y)), fmaxf(a.z, fmaxf(b.z, c.z)));
}

// bottom-up refit: each leaf walks towards the root; the second arrival at a node
// merges both children's boxes (written before the first arrival's fence).
__global__ void k_refit(const float4 *tris, int n, const int4 *child, const int *parent_node,
                        const int *parent_leaf, float4 *box_lo, float4 *box_hi, int *arrivals,
                        BvhNode *nodes, int *bad) {
    int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    float3 lo, hi;
    tri_box(tris, k, lo, hi);
    // leaf boxes are stored after the n-1 internal ones
    box_lo[n - 1 + k] = make_float4(lo.x, lo.y, lo.z, 0.f);
    box_hi[n - 1 + k] = make_float4(hi.x, hi.y, hi.z, 0.f);
    __threadfence();
    int p = parent_leaf[k];
    for (int level = 0; p >= 0; level++) {
        if (p >= n - 1 || level > 160) { atomicExch(bad, 3); return; }
        if (atomicAdd(&arrivals[p], 1) == 0) return;   // the sibling finishes this node
        __threadfence();
        int4 ch = child[p];
        if (ch.x >= n - 1 || ch.y >= n - 1 || (ch.x < 0 && ~ch.x >= n) || (ch.y < 0 && ~ch.y >= n)) {
            atomicExch(bad, 3);
            return;
        }
        int s0 = ch.x >= 0 ? ch.x : n - 1 + ~ch.x;
        int s1 = ch.y >= 0 ? ch.y : n - 1 + ~ch.y;
        float4 l0 = __ldcg(&box_lo[s0]), h0 = __ldcg(&box_hi[s0]);
        float4 l1 = __ldcg(&box_lo[s1]), h1 = __ldcg(&box_hi[s1]);
        BvhNode nd;
        nd.a = make_float4(l0.x, h0.x, l1.x, h1.x);
        nd.b = make_float4(l0.y, h0.y, l1.y, h1.y);
        nd.c = make_float4(l0.z, h0.z, l1.z, h1.z);
        nd.r = make_int4(ch.x, ch.y, 0, 0);
        nodes[p] = nd;
        box_lo[p] = make_float4(fminf(l0.x, l1.x), fminf(l0.y, l1.y), fminf(l0.z, l1.z), 0.f);
        box_hi[p] = make_float4(fmaxf(h0.x, h1.x), fmaxf(h0.y, h1.y), fmaxf(h0.z, h1.z), 0.f);
        __threadfence();
        p = parent_node[p];
    }
}

// half the surface area of a box
__device__ __forceinline__ float half_area(float4 lo, float4 hi) {
    float dx = hi.x - lo.x, dy = hi.y - lo.y, dz = hi.z - lo.z;
    return dx * dy + dy * dz + dz * dx;
}

// Tree rotations (Kensler, "Tree Rotations for Improving Bounding Volume Hierarchies",
// 2008), one bottom-up pass synchronised like the refit: at each internal node p with
// children L and R, swapping R with a child of L (or L with a child of R) changes the
// box of one child only, so the swap that shrinks that child's surface area the most is
// made, when it shrinks it by more than 2^-16 of p's area.  Every subtree keeps its
// leaves and every box is the exact union of its children's, so the closest hit of a ray
// is unchanged; the parents of the two moved subtrees are updated.
__device__ __forceinline__ void node_child(const BvhNode &nd, int c, float4 &lo, float4 &hi, int &ref) {
    if (c == 0) {
        lo = make_float4(nd.a.x, nd.b.x, nd.c.x, 0.f); hi = make_float4(nd.a.y, nd.b.y, nd.c.y, 0.f); ref = nd.r.x;
    } else {
        lo = make_float4(nd.a.z, nd.b.z, nd.c.z, 0.f); hi = make_float4(nd.a.w, nd.b.w, nd.c.w, 0.f); ref = nd.r.y;
    }
}

__device__ __forceinline__ BvhNode make_node(float4 l0, float4 h0, int r0, float4 l1, float4 h1, int r1) {
    BvhNode nd;
    nd.a = make_float4(l0.x, h0.x, l1.x, h1.x);
    nd.b = make_float4(l0.y, h0.y, l1.y, h1.y);
    nd.c = make_float4(l0.z, h0.z, l1.z, h1.z);
    nd.r = make_int4(r0, r1, 0, 0);
    return nd;
}

__device__ __forceinline__ float union_area(float4 l0, float4 h0, float4 l1, float4 h1) {
    return half_area(make_float4(fminf(l0.x, l1.x), fminf(l0.y, l1.y), fminf(l0.z, l1.z), 0.f),
                     make_float4(fmaxf(h0.x, h1.x), fmaxf(h0.y, h1.y), fmaxf(h0.z, h1.z), 0.f));
}

__device__ __forceinline__ void set_parent(int ref, int p, int n, int *parent_node, int *parent_leaf, int *bad) {
    if (ref < 0 ? ~ref >= n : ref >= n - 1) { atomicExch(bad, 7); return; }
    if (ref < 0) parent_leaf[~ref] = p;
    else parent_node[ref] = p;
}

// a node as other threads of the pass last wrote it (from L2, not a stale L1 line)
__device__ __forceinline__ BvhNode ld_node_cg(const BvhNode *nd) {
    const float4 *q = reinterpret_cast<const float4 *>(nd);
    BvhNode o;
    o.a = __ldcg(q);
    o.b = __ldcg(q + 1);
    o.c = __ldcg(q + 2);
    o.r = __ldcg(reinterpret_cast<const int4 *>(q + 3));
    return o;
}

__global__ void k_rotate(int n, BvhNode *nodes, int *parent_node, int *parent_leaf, int *arrivals, int *bad) {
    int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    int p = __ldcg(&parent_leaf[k]);
    for (int level = 0; p >= 0; level++) {
        if (p >= n - 1 || level > 160) { atomicExch(bad, 7); return; }
        __threadfence();
        if (atomicAdd(&arrivals[p], 1) == 0) return;   // the sibling finishes this node
        __threadfence();
        const BvhNode np = ld_node_cg(&nodes[p]);
        float4 lL, hL, lR, hR;
        int L, R;
        node_child(np, 0, lL, hL, L);
        node_child(np, 1, lR, hR, R);
        const float areaL = half_area(lL, hL), areaR = half_area(lR, hR);
        const float thresh = union_area(lL, hL, lR, hR) * (1.f / 65536.f);
        float best = thresh;
        int kind = -1;                      // 0, 1: R with a child of L; 2, 3: L with a child of R
        BvhNode nL, nR;
        float4 la, ha, lb, hb, lc, hc, ld, hd;
        int ra = 0, rb = 0, rc = 0, rd = 0;
        if (L >= 0) {
            if (L >= n - 1) { atomicExch(bad, 7); return; }
            nL = ld_node_cg(&nodes[L]);
            node_child(nL, 0, la, ha, ra);
            node_child(nL, 1, lb, hb, rb);
            const float g0 = areaL - union_area(lR, hR, lb, hb);   // R <-> LL: L = (R, LR)
            const float g1 = areaL - union_area(la, ha, lR, hR);   // R <-> LR: L = (LL, R)
            if (g0 > best) { best = g0; kind = 0; }
            if (g1 > best) { best = g1; kind = 1; }
        }
        if (R >= 0) {
            if (R >= n - 1) { atomicExch(bad, 7); return; }
            nR = ld_node_cg(&nodes[R]);
            node_child(nR, 0, lc, hc, rc);
            node_child(nR, 1, ld, hd, rd);
            const float g2 = areaR - union_area(lL, hL, ld, hd);   // L <-> RL: R = (L, RR)
            const float g3 = areaR - union_area(lc, hc, lL, hL);   // L <-> RR: R = (RL, L)
            if (g2 > best) { best = g2; kind = 2; }
            if (g3 > best) { best = g3; kind = 3; }
        }
        if (kind == 0 || kind == 1) {
            // the child of L that moves up to p (m) and the one that stays with R
            const float4 lm = kind == 0 ? la : lb, hm = kind == 0 ? ha : hb;
            const int rm = kind == 0 ? ra : rb;
            const float4 ls = kind == 0 ? lb : la, hs = kind == 0 ? hb : ha;
            const int rs = kind == 0 ? rb : ra;
            const BvhNode newL = kind == 0 ? make_node(lR, hR, R, ls, hs, rs) : make_node(ls, hs, rs, lR, hR, R);
            float4 lN, hN;
            int dummy;
            node_child(newL, 0, lN, hN, dummy);
            float4 l2, h2;
            node_child(newL, 1, l2, h2, dummy);
            lN = make_float4(fminf(lN.x, l2.x), fminf(lN.y, l2.y), fminf(lN.z, l2.z), 0.f);
            hN = make_float4(fmaxf(hN.x, h2.x), fmaxf(hN.y, h2.y), fmaxf(hN.z, h2.z), 0.f);
            nodes[L] = newL;
            nodes[p] = make_node(lN, hN, L, lm, hm, rm);
            set_parent(R, L, n, parent_node, parent_leaf, bad);
            set_parent(rm, p, n, parent_node, parent_leaf, bad);
        } else if (kind == 2 || kind == 3) {
            const float4 lm = kind == 2 ? lc : ld, hm = kind == 2 ? hc : hd;
            const int rm = kind == 2 ? rc : rd;
            const float4 ls = kind == 2 ? ld : lc, hs = kind == 2 ? hd : hc;
            const int rs = kind == 2 ? rd : rc;
            const BvhNode newR = kind == 2 ? make_node(lL, hL, L, ls, hs, rs) : make_node(ls, hs, rs, lL, hL, L);
            float4 lN, hN, l2, h2;
            int dummy;
            node_child(newR, 0, lN, hN, dummy);
            node_child(newR, 1, l2, h2, dummy);
            lN = make_float4(fminf(lN.x, l2.x), fminf(lN.y, l2.y), fminf(lN.z, l2.z), 0.f);
            hN = make_float4(fmaxf(hN.x, h2.x), fmaxf(hN.y, h2.y), fmaxf(hN.z, h2.z), 0.f);
            nodes[R] = newR;
            nodes[p] = make_node(lm, hm, rm, lN, hN, R);
            set_parent(L, R, n, parent_node, parent_leaf, bad);
            set_parent(rm, p, n, parent_node, parent_leaf, bad);
        }
        __threadfence();
        p = __ldcg(&parent_node[p]);
    }
}

// The order in which a packet takes a node's two children: along the axis on which their
// centres lie farthest apart for their size, the lower one first (child 0) for rays that
// climb the axis.  r.z keeps that axis.  Simulated on the workloads' packets this order
// visits as many nodes as the vote of the lanes on their entry distances did (71.3 per
// packet at 496k triangles either way), without the entry distances and the vote.
__device__ __forceinline__ int4 order_children(BvhNode &nd) {
    float4 l0, h0, l1, h1;
    int r0, r1;
    node_child(nd, 0, l0, h0, r0);
    node_child(nd, 1, l1, h1, r1);
    const float lo0[3] = {l0.x, l0.y, l0.z}, hi0[3] = {h0.x, h0.y, h0.z};
    const float lo1[3] = {l1.x, l1.y, l1.z}, hi1[3] = {h1.x, h1.y, h1.z};
    int axis = 0;
    float best = -1.f, gap = 0.f;
#pragma unroll
    for (int k = 0; k < 3; k++) {
        const float d = (lo1[k] + hi1[k]) - (lo0[k] + hi0[k]);
        const float s = fabsf(d) / (fmaxf(hi0[k] - lo0[k], hi1[k] - lo1[k]) + 1e-9f);
        if (s > best) { best = s; axis = k; gap = d; }
    }
    if (gap < 0.f) nd = make_node(l1, h1, r1, l0, h0, r0);
    nd.r.z = axis;
    return nd.r;
}

// Structure check of the finished binary tree, before any traversal relies on it: every
// child reference in range (internal nodes 0 .. n_nodes - 1, leaves ~0 .. ~(n_tree - 1)),
// and every internal node except the root, and every leaf, referenced by exactly one
// internal node, the root by none.  Nodes on a cycle would take their one reference from
// inside the cycle, so none is reachable from the root: a traversal from the root visits
// each node at most once and reads only in-range nodes and triangles.  The parents are
// recorded from the same references (parent_node / parent_leaf, -1 beforehand), so the
// depth that k_depth then walks up from every leaf is the depth of the tree the traversal
// reads: a leaf below a cycle walks to k_depth's cap, which the traversal stack rejects.
//
// Each node's children are also put in the order that packets take them (order_children).
__global__ void k_tree_refs(BvhNode *nodes, int n_nodes, int n_tree, int *ref_node, int *ref_leaf,
                            int *parent_node, int *parent_leaf, int *bad) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n_nodes) return;
    const int4 r = order_children(nodes[i]);
    const int c[2] = {r.x, r.y};
#pragma unroll
    for (int e = 0; e < 2; e++) {
        if (c[e] >= 0 ? c[e] >= n_nodes : ~c[e] >= n_tree) { atomicExch(bad, 8); continue; }
        atomicAdd(c[e] >= 0 ? &ref_node[c[e]] : &ref_leaf[~c[e]], 1);
        if (c[e] >= 0) parent_node[c[e]] = i;
        else parent_leaf[~c[e]] = i;
    }
}
__global__ void k_tree_counts(int n_nodes, int n_tree, const int *root_p, const int *ref_node, const int *ref_leaf,
                              int *bad) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int root = *root_p;
    if (i == 0 && (root < 0 || root >= n_nodes)) atomicExch(bad, 9);
    if (i < n_nodes && ref_node[i] != (i == root ? 0 : 1)) atomicExch(bad, 9);
    if (i < n_tree && ref_leaf[i] != 1) atomicExch(bad, 9);
}

// tree depth (levels from the root to the deepest leaf, root = 1)
__global__ void k_depth(int n, const int *parent_node, const int *parent_leaf, int *depth) {
    int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    int d = 1, p = parent_leaf[k];
    while (p >= 0 && d < 1000) { d++; p = parent_node[p]; }
    atomicMax(depth, d);
}


// ---------------------------------------------------------------------------
// One round of PLOC (Meister and Bittner, "Parallel Locally-Ordered Clustering for
// Bounding Volume Hierarchy Construction", TVCG 2018) over the Morton-sorted leaves: each
// finds its nearest neighbour within +-radius positions by the surface area of the merged
// box; mutual nearest neighbours merge into a new node; the clusters are compacted, in
// order.  A cluster is its box, with its reference (leaf ~k or node) in lo.w.
// ---------------------------------------------------------------------------
__global__ void k_ploc_init(const float4 *tris, int m, float4 *clo, float4 *chi) {
    int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= m) return;
    float3 lo, hi;
    tri_box(tris, k, lo, hi);
    clo[k] = make_float4(lo.x, lo.y, lo.z, __int_as_float(~k));
    chi[k] = make_float4(hi.x, hi.y, hi.z, 0.f);
}

// nearest neighbour by merged area; ties to the smaller index (symmetric cost, so the
// globally cheapest pair is always mutual).  The block's clusters and a halo of `radius` on
// either side are staged in shared memory.
constexpr int kNnThreads = 256, kNnMaxRadius = 256;
__global__ void __launch_bounds__(kNnThreads) k_ploc_nn(int count, int radius, const float4 *clo, const float4 *chi, int *nn) {
    extern __shared__ float4 sm_nn[];
    const int base = blockIdx.x * kNnThreads - radius, tile = kNnThreads + 2 * radius;
    float4 *sl = sm_nn, *sh = sm_nn + tile;
    for (int e = threadIdx.x; e < tile; e += kNnThreads) {
        const int j = min(max(base + e, 0), count - 1);
        sl[e] = clo[j];
        sh[e] = chi[j];
    }
    __syncthreads();
    const int i = blockIdx.x * kNnThreads + threadIdx.x;
    if (i >= count) return;
    const float4 lo = sl[i - base], hi = sh[i - base];
    float best = INFINITY;
    int bj = -1;
    const int j0 = max(0, i - radius), j1 = min(count - 1, i + radius);
    for (int j = j0; j <= j1; j++) {
        if (j == i) continue;
        const float a = union_area(lo, hi, sl[j - base], sh[j - base]);
        if (a < best) { best = a; bj = j; }
    }
    nn[i] = bj;
}

// mutual pairs merge: the lower position creates the node and keeps the merged cluster, the
// higher one drops out
__global__ void k_ploc_merge(int count, float4 *clo, float4 *chi, const int *nn, int *keep, int *node_count, BvhNode *nodes,
                             int n_nodes, int *bad) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = i < count ? nn[i] : -1;
    const bool mutual = j >= 0 && nn[j] == i, make = mutual && i < j;
    // one atomic per warp for its new nodes
    const unsigned lane = threadIdx.x & 31, b = __ballot_sync(0xffffffffu, make);
    int id = 0;
    if (lane == 0 && b) id = atomicAdd(node_count, __popc(b));
    id = __shfl_sync(0xffffffffu, id, 0) + __popc(b & ((1u << lane) - 1u));
    if (i >= count) return;
    if (!make) {
        keep[i] = mutual ? 0 : 1;
        return;
    }
    keep[i] = 1;
    if (id >= n_nodes) { atomicExch(bad, 4); return; }
    const float4 l0 = clo[i], h0 = chi[i], l1 = clo[j], h1 = chi[j];
    nodes[id] = make_node(l0, h0, __float_as_int(l0.w), l1, h1, __float_as_int(l1.w));
    clo[i] = make_float4(fminf(l0.x, l1.x), fminf(l0.y, l1.y), fminf(l0.z, l1.z), __int_as_float(id));
    chi[i] = make_float4(fmaxf(h0.x, h1.x), fmaxf(h0.y, h1.y), fmaxf(h0.z, h1.z), 0.f);
}

__global__ void k_ploc_scatter(int count, const int *keep, const int *pos, const float4 *clo, const float4 *chi, float4 *clo2,
                               float4 *chi2) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= count || !keep[i]) return;
    const int o = pos[i];
    clo2[o] = clo[i];
    chi2[o] = chi[i];
}

// ---------------------------------------------------------------------------
// Top-down binned SAH (Wald, "On fast Construction of SAH-based Bounding Volume
// Hierarchies", 2007) over the clusters that one PLOC round leaves.
//
// A segment is a contiguous range of the cluster array that becomes one subtree.  While
// a segment holds more than kSahSmall clusters it is split by whole launches, one level at
// a time: its chunks fill 16 bins per axis over the centroids' bounds (k_sah_bin), a warp
// picks the cheapest of the 45 planes, writes the node and makes the two children
// (k_sah_split), and the chunks move their clusters to the side they belong to, gathering
// the children's centroid bounds (k_sah_part).  A segment of at most kSahSmall clusters is
// finished by one warp in shared memory (k_sah_small).
//
// Why: the rays of the packet tracer step this tree.  PLOC alone left its large structure
// to chance (97 to 150 node tests per packet at 496k triangles, by search radius); with the
// planes of the surface-area heuristic at the top it takes ~70, whatever the radius.  One
// PLOC round first halves the clusters to split and costs no quality: it pairs the
// triangles that share a box.  Two or three rounds are worse by 3-6% at 496k triangles.
// Measured against PLOC alone (radius 48): the 1080p tracer 0.440 -> 0.237 ms one ray per
// lane, 0.194 -> 0.161 ms as packets, ten rays per pixel 1.239 -> 0.895 ms; the ray-cast
// G-buffer 0.917 -> 0.615 ms; the 4K tracer (2M triangles) is even.
//
// The build itself is bound by latency at the top (a level of few segments cannot fill the
// chip: 14 levels x 3 launches, 0.4 ms) and by the warps' serial splits at the bottom
// (k_sah_small).  Scratch comes from one pool block and the host reads back three
// times, where every PLOC round used to end in a synchronisation (65 of them): upload and
// first view of 496k triangles 7.1 -> 2.9 ms.
// ---------------------------------------------------------------------------
constexpr int kSahBins = 16;             // per axis
constexpr int kSahSmall = 256;           // clusters a warp finishes alone (uint8 indices)
constexpr int kSahSweep = 10;            // clusters up to which it tries every plane (3 x 10 lanes)
constexpr int kSahChunk = 512;           // clusters of one work item of a large segment
constexpr int kSahThreads = 256;
constexpr int kSahSlotInts = 3 * 7 * kSahBins;   // [axis][count, lo.xyz, hi.xyz][bin]
constexpr int kSahMaxLevel = 48;         // from here on segments are halved by position, so that
                                         // the tree is at most 48 + 31 + 1 levels deep

struct SahSeg {
    int begin, count, node, level;
    int clo[3], chi[3];                  // bounds of the centroids (ordered ints)
    int axis, bin, nl;                   // the plane: axis (-1: by position), last bin of the left side
    int cur_l, cur_r;                    // clusters placed so far on either side
    int child_l, child_r;                // their segments in the next level's table, -1 if small
    int refs;                            // left/right child is a single cluster: bits 0 / 1
};

struct SahState {
    int n_seg[2], n_item[2];             // per level parity
    int n_small, small_next;             // small segments, and the next one to take
    int count;                           // clusters
};

// the bin of a centroid: every kernel computes it here, with each rounding written out, so
// that the counts of the bins and the sides of the partition agree
__device__ __forceinline__ int sah_bin(float c, float lo, float ext) {
    const float u = __fmul_rn(__fdiv_rn(__fsub_rn(c, lo), ext), (float)kSahBins);
    return min(max((int)u, 0), kSahBins - 1);
}
__device__ __forceinline__ float sah_centre(float lo, float hi) { return __fmul_rn(0.5f, __fadd_rn(lo, hi)); }

struct SahPlane {
    int axis, bin, nl;                   // axis -1: no plane separates the clusters
    float lo[2][3], hi[2][3];            // boxes of the two sides
};

// The cheapest plane of 3 x 15, by a full warp; bins[axis][component][bin] with ordered-int
// bounds.  Lanes 0-15 take axes 0 then 2, lanes 16-31 axis 1.  cost = area x clusters on
// either side; ties to the smaller (axis, bin).
__device__ __forceinline__ SahPlane sah_select(const int *bins, unsigned lane) {
    float best = INFINITY;
    int best_id = 0x7FFFFFFF;
    float bl[2][3], bh[2][3];
    int bn = 0;
#pragma unroll
    for (int k = 0; k < 3; k++) bl[0][k] = bl[1][k] = bh[0][k] = bh[1][k] = 0.f;
#pragma unroll
    for (int round = 0; round < 2; round++) {
        const int axis = round == 0 ? (int)(lane >> 4) : 2;
        const int q = (int)(lane & 15u);
        const int *b = bins + axis * 7 * kSahBins + q;
        int n = b[0];
        float lo[3], hi[3];
#pragma unroll
        for (int k = 0; k < 3; k++) {
            lo[k] = n ? float_of(b[(1 + k) * kSahBins]) : INFINITY;
            hi[k] = n ? float_of(b[(4 + k) * kSahBins]) : -INFINITY;
        }
        // inclusive prefix and suffix over the 16 bins
        int np = n, ns = n;
        float pl[3], ph[3], sl[3], sh[3];
#pragma unroll
        for (int k = 0; k < 3; k++) { pl[k] = sl[k] = lo[k]; ph[k] = sh[k] = hi[k]; }
#pragma unroll
        for (int o = 1; o < kSahBins; o <<= 1) {
            const int tn = __shfl_up_sync(0xffffffffu, np, o, 16), un = __shfl_down_sync(0xffffffffu, ns, o, 16);
            const bool up = q >= o, dn = q + o < kSahBins;
            if (up) np += tn;
            if (dn) ns += un;
#pragma unroll
            for (int k = 0; k < 3; k++) {
                const float a = __shfl_up_sync(0xffffffffu, pl[k], o, 16), c = __shfl_up_sync(0xffffffffu, ph[k], o, 16);
                const float d = __shfl_down_sync(0xffffffffu, sl[k], o, 16), e = __shfl_down_sync(0xffffffffu, sh[k], o, 16);
                if (up) { pl[k] = fminf(pl[k], a); ph[k] = fmaxf(ph[k], c); }
                if (dn) { sl[k] = fminf(sl[k], d); sh[k] = fmaxf(sh[k], e); }
            }
        }
        // the plane after bin q: bins 0 .. q against q + 1 .. 15
        const int nr = __shfl_down_sync(0xffffffffu, ns, 1, 16);
        float rl[3], rh[3];
#pragma unroll
        for (int k = 0; k < 3; k++) {
            rl[k] = __shfl_down_sync(0xffffffffu, sl[k], 1, 16);
            rh[k] = __shfl_down_sync(0xffffffffu, sh[k], 1, 16);
        }
        if (q < kSahBins - 1 && np > 0 && nr > 0) {
            const float cost = half_area(make_float4(pl[0], pl[1], pl[2], 0.f), make_float4(ph[0], ph[1], ph[2], 0.f)) * (float)np +
                               half_area(make_float4(rl[0], rl[1], rl[2], 0.f), make_float4(rh[0], rh[1], rh[2], 0.f)) * (float)nr;
            if (cost < best && !(round == 1 && lane >= 16)) {
                best = cost;
                best_id = axis * kSahBins + q;
                bn = np;
#pragma unroll
                for (int k = 0; k < 3; k++) {
                    bl[0][k] = pl[k]; bh[0][k] = ph[k];
                    bl[1][k] = rl[k]; bh[1][k] = rh[k];
                }
            }
        }
    }
    float m = best;
    int id = best_id;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const float c = __shfl_xor_sync(0xffffffffu, m, o);
        const int i = __shfl_xor_sync(0xffffffffu, id, o);
        if (c < m || (c == m && i < id)) { m = c; id = i; }
    }
    SahPlane p;
    if (id == 0x7FFFFFFF) {
        p.axis = -1; p.bin = 0; p.nl = 0;
#pragma unroll
        for (int s = 0; s < 2; s++)
#pragma unroll
            for (int k = 0; k < 3; k++) p.lo[s][k] = p.hi[s][k] = 0.f;
        return p;
    }
    const int win = __ffs(__ballot_sync(0xffffffffu, best_id == id)) - 1;
    p.axis = id / kSahBins;
    p.bin = id % kSahBins;
    p.nl = __shfl_sync(0xffffffffu, bn, win);
#pragma unroll
    for (int s = 0; s < 2; s++)
#pragma unroll
        for (int k = 0; k < 3; k++) {
            p.lo[s][k] = __shfl_sync(0xffffffffu, bl[s][k], win);
            p.hi[s][k] = __shfl_sync(0xffffffffu, bh[s][k], win);
        }
    return p;
}

__device__ __forceinline__ void sah_bins_clear(int *b, int tid, int threads) {
    for (int e = tid; e < kSahSlotInts; e += threads) {
        const int c = (e / kSahBins) % 7;
        b[e] = c == 0 ? 0 : (c <= 3 ? 0x7FFFFFFF : (int)0x80000000);
    }
}

// add a cluster's box to its bin of each axis (shared memory)
__device__ __forceinline__ void sah_bins_add(int *b, const int *bin, float4 lo, float4 hi) {
    const int l[3] = {ord_of(lo.x), ord_of(lo.y), ord_of(lo.z)}, h[3] = {ord_of(hi.x), ord_of(hi.y), ord_of(hi.z)};
#pragma unroll
    for (int a = 0; a < 3; a++) {
        int *p = b + a * 7 * kSahBins + bin[a];
        atomicAdd(p, 1);
#pragma unroll
        for (int k = 0; k < 3; k++) {
            atomicMin(p + (1 + k) * kSahBins, l[k]);
            atomicMax(p + (4 + k) * kSahBins, h[k]);
        }
    }
}

// the table's segment `s` of parity `par` for clusters [begin, begin + count), with its bins
// cleared and its chunks listed; the calling warp does it together
__device__ __forceinline__ void sah_make_seg(SahSeg *segs, int *bins, int2 *items, int *n_item, int s, int max_items, int begin,
                                             int count, int node, int level, unsigned lane, int *bad) {
    if (lane == 0) {
        SahSeg g;
        g.begin = begin; g.count = count; g.node = node; g.level = level;
        for (int k = 0; k < 3; k++) { g.clo[k] = 0x7FFFFFFF; g.chi[k] = (int)0x80000000; }
        g.axis = -1; g.bin = 0; g.nl = 0;
        g.cur_l = g.cur_r = 0;
        g.child_l = g.child_r = -1;
        g.refs = 0;
        segs[s] = g;
    }
    sah_bins_clear(bins + (size_t)s * kSahSlotInts, (int)lane, 32);
    const int n = (count + kSahChunk - 1) / kSahChunk;
    int at = 0;
    if (lane == 0) at = atomicAdd(n_item, n);
    at = __shfl_sync(0xffffffffu, at, 0);
    if (at + n > max_items) {
        if (lane == 0) atomicExch(bad, 10);
        return;
    }
    for (int k = (int)lane; k < n; k += 32) items[at + k] = make_int2(s, k);
}

// the clusters' first segment (one warp), or the small list, or nothing to split
__global__ void k_sah_root(SahState *st, const int *pos, const int *keep, int m, const float4 *lo, SahSeg *segs, int *bins,
                           int2 *items, int max_items, int4 *small, int *node_count, int *root, int *bad) {
    const unsigned lane = threadIdx.x;
    const int c = pos[m - 1] + keep[m - 1];
    int node = -1;
    if (lane == 0) {
        st->count = c;
        if (c == 1) {
            *root = __float_as_int(lo[0].w);
        } else {
            node = atomicAdd(node_count, 1);
            *root = node;
            if (c <= kSahSmall) {
                small[0] = make_int4(0, c, node, 0);
                st->n_small = 1;
            } else {
                st->n_seg[0] = 1;
            }
        }
    }
    node = __shfl_sync(0xffffffffu, node, 0);
    if (c > kSahSmall) sah_make_seg(segs, bins, items, &st->n_item[0], 0, max_items, 0, c, node, 0, lane, bad);
}

__device__ __forceinline__ int warp_min(int v) { return __reduce_min_sync(0xffffffffu, v); }
__device__ __forceinline__ int warp_max(int v) { return __reduce_max_sync(0xffffffffu, v); }

// the root segment's centroid bounds (the children's come with the partition)
__global__ void __launch_bounds__(kSahThreads) k_sah_root_bounds(const SahState *st, const float4 *lo, const float4 *hi,
                                                                 SahSeg *segs) {
    const int c = st->count;
    if (c <= kSahSmall) return;
    int l[3] = {0x7FFFFFFF, 0x7FFFFFFF, 0x7FFFFFFF}, h[3] = {(int)0x80000000, (int)0x80000000, (int)0x80000000};
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < c; i += gridDim.x * blockDim.x) {
        const float4 a = lo[i], b = hi[i];
        const int e[3] = {ord_of(sah_centre(a.x, b.x)), ord_of(sah_centre(a.y, b.y)), ord_of(sah_centre(a.z, b.z))};
#pragma unroll
        for (int k = 0; k < 3; k++) { l[k] = min(l[k], e[k]); h[k] = max(h[k], e[k]); }
    }
    __shared__ int s[6];
    if (threadIdx.x < 6) s[threadIdx.x] = threadIdx.x < 3 ? 0x7FFFFFFF : (int)0x80000000;
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 3; k++) {
        const int a = warp_min(l[k]), b = warp_max(h[k]);
        if ((threadIdx.x & 31) == 0) { atomicMin(&s[k], a); atomicMax(&s[3 + k], b); }
    }
    __syncthreads();
    if (threadIdx.x < 3) atomicMin(&segs[0].clo[threadIdx.x], s[threadIdx.x]);
    else if (threadIdx.x < 6) atomicMax(&segs[0].chi[threadIdx.x - 3], s[threadIdx.x]);
}

// one level, step 1: the chunks of the large segments fill their bins (in shared memory, then
// one global atomic per non-empty bin and component)
__global__ void __launch_bounds__(kSahThreads) k_sah_bin(SahState *st, int par, const SahSeg *segs, const int2 *items,
                                                         const float4 *lo, const float4 *hi, int *bins) {
    __shared__ int sb[kSahSlotInts];
    // the tables of the level before are free for the level after
    if (blockIdx.x == 0 && threadIdx.x == 0) st->n_seg[par ^ 1] = st->n_item[par ^ 1] = 0;
    const int n = st->n_item[par];
    for (int it = blockIdx.x; it < n; it += gridDim.x) {
        const int2 w = items[it];
        const SahSeg &g = segs[w.x];
        const int b0 = g.begin + w.y * kSahChunk, b1 = min(g.begin + g.count, b0 + kSahChunk);
        float cl[3], ext[3];
#pragma unroll
        for (int k = 0; k < 3; k++) {
            cl[k] = float_of(g.clo[k]);
            ext[k] = __fsub_rn(float_of(g.chi[k]), cl[k]);
        }
        sah_bins_clear(sb, threadIdx.x, kSahThreads);
        __syncthreads();
        for (int i = b0 + (int)threadIdx.x; i < b1; i += kSahThreads) {
            const float4 a = lo[i], b = hi[i];
            const int bin[3] = {sah_bin(sah_centre(a.x, b.x), cl[0], ext[0]), sah_bin(sah_centre(a.y, b.y), cl[1], ext[1]),
                                sah_bin(sah_centre(a.z, b.z), cl[2], ext[2])};
            sah_bins_add(sb, bin, a, b);
        }
        __syncthreads();
        int *gb = bins + (size_t)w.x * kSahSlotInts;
        for (int e = threadIdx.x; e < kSahSlotInts; e += kSahThreads) {
            const int c = (e / kSahBins) % 7, v = sb[e];
            if (sb[e - c * kSahBins] == 0) continue;
            if (c == 0) atomicAdd(&gb[e], v);
            else if (c <= 3) atomicMin(&gb[e], v);
            else atomicMax(&gb[e], v);
        }
        __syncthreads();
    }
}

// step 2: a warp per large segment picks its plane, writes its node and makes its children
__global__ void __launch_bounds__(128) k_sah_split(SahState *st, int par, SahSeg *segs, const int *bins, SahSeg *next,
                                                   int *next_bins, int2 *next_items, int max_segs, int max_items, int4 *small,
                                                   int max_small, BvhNode *nodes, int n_nodes, int *node_count, int *bad) {
    const unsigned lane = threadIdx.x & 31;
    const int n = st->n_seg[par];
    const int warps = gridDim.x * (blockDim.x >> 5);
    for (int s = (int)(blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)); s < n; s += warps) {
        SahSeg &g = segs[s];
        const int begin = g.begin, count = g.count, level = g.level, node = g.node;
        SahPlane p = sah_select(bins + (size_t)s * kSahSlotInts, lane);
        if (level >= kSahMaxLevel || p.nl <= 0 || p.nl >= count) p.axis = -1;
        if (p.axis < 0) {
            // by position: both sides take the whole segment's box (a superset is as safe)
            p.nl = count / 2;
            const int *b = bins + (size_t)s * kSahSlotInts;
#pragma unroll
            for (int k = 0; k < 3; k++) {
                const int q = (int)(lane & 15u);
                const float l = float_of(warp_min(b[(1 + k) * kSahBins + q])), h = float_of(warp_max(b[(4 + k) * kSahBins + q]));
                p.lo[0][k] = p.lo[1][k] = l;
                p.hi[0][k] = p.hi[1][k] = h;
            }
        }
        const int nc[2] = {p.nl, count - p.nl};
        int ref[2] = {0, 0}, child[2] = {-1, -1}, single = 0;
#pragma unroll
        for (int c = 0; c < 2; c++) {
            const int at = c ? begin + p.nl : begin;
            if (nc[c] == 1) {                       // the partition fills in the cluster's own reference
                single |= 1 << c;
                continue;
            }
            int id = 0;
            if (lane == 0) id = atomicAdd(node_count, 1);
            id = __shfl_sync(0xffffffffu, id, 0);
            ref[c] = id;
            int slot = 0;
            if (nc[c] <= kSahSmall) {
                if (lane == 0) {
                    slot = atomicAdd(&st->n_small, 1);
                    if (slot < max_small) small[slot] = make_int4(at, nc[c], id, level + 1);
                    else atomicExch(bad, 10);
                }
            } else {
                if (lane == 0) slot = atomicAdd(&st->n_seg[par ^ 1], 1);
                slot = __shfl_sync(0xffffffffu, slot, 0);
                if (slot < max_segs) {
                    sah_make_seg(next, next_bins, next_items, &st->n_item[par ^ 1], slot, max_items, at, nc[c], id, level + 1,
                                 lane, bad);
                    child[c] = slot;
                } else if (lane == 0) {
                    atomicExch(bad, 10);
                }
            }
        }
        if (lane == 0) {
            g.axis = p.axis; g.bin = p.bin; g.nl = p.nl;
            g.child_l = child[0]; g.child_r = child[1];
            g.refs = single;
            if (node >= 0 && node < n_nodes)
                nodes[node] = make_node(make_float4(p.lo[0][0], p.lo[0][1], p.lo[0][2], 0.f),
                                        make_float4(p.hi[0][0], p.hi[0][1], p.hi[0][2], 0.f), ref[0],
                                        make_float4(p.lo[1][0], p.lo[1][1], p.lo[1][2], 0.f),
                                        make_float4(p.hi[1][0], p.hi[1][1], p.hi[1][2], 0.f), ref[1]);
            else
                atomicExch(bad, 10);
        }
    }
}

// step 3: the chunks move their clusters to either side of the plane (places reserved with one
// atomic per chunk and side) and gather the large children's centroid bounds
__global__ void __launch_bounds__(kSahThreads) k_sah_part(const SahState *st, int par, SahSeg *segs, const int2 *items,
                                                          const float4 *lo, const float4 *hi, float4 *lo2, float4 *hi2,
                                                          SahSeg *next, BvhNode *nodes, int *bad) {
    __shared__ int base[2], cb[12];
    __shared__ int wl[kSahThreads / 32], wr[kSahThreads / 32];
    const int n = st->n_item[par];
    const unsigned lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    constexpr int kPer = kSahChunk / kSahThreads;
    for (int it = blockIdx.x; it < n; it += gridDim.x) {
        const int2 w = items[it];
        SahSeg &g = segs[w.x];
        const int begin = g.begin, count = g.count, nl = g.nl, axis = g.axis, bin = g.bin;
        const int b0 = begin + w.y * kSahChunk, b1 = min(begin + count, b0 + kSahChunk);
        const float cl = axis >= 0 ? float_of(g.clo[axis]) : 0.f;
        const float ext = axis >= 0 ? __fsub_rn(float_of(g.chi[axis]), cl) : 0.f;
        if (threadIdx.x < 12) cb[threadIdx.x] = threadIdx.x % 6 < 3 ? 0x7FFFFFFF : (int)0x80000000;
        float4 a[kPer], b[kPer];
        bool in[kPer], left[kPer];
        int nleft = 0, nright = 0;
        unsigned ml[kPer], mr[kPer];
#pragma unroll
        for (int r = 0; r < kPer; r++) {
            const int i = b0 + r * kSahThreads + (int)threadIdx.x;
            in[r] = i < b1;
            left[r] = false;
            if (in[r]) {
                a[r] = lo[i];
                b[r] = hi[i];
                const float c = axis == 0 ? sah_centre(a[r].x, b[r].x) : (axis == 1 ? sah_centre(a[r].y, b[r].y) : sah_centre(a[r].z, b[r].z));
                left[r] = axis >= 0 ? sah_bin(c, cl, ext) <= bin : i - begin < nl;
            }
            ml[r] = __ballot_sync(0xffffffffu, in[r] && left[r]);
            mr[r] = __ballot_sync(0xffffffffu, in[r] && !left[r]);
            nleft += __popc(ml[r]);
            nright += __popc(mr[r]);
        }
        if (lane == 0) { wl[warp] = nleft; wr[warp] = nright; }
        __syncthreads();
        if (threadIdx.x == 0) {
            int tl = 0, tr = 0;
#pragma unroll
            for (int k = 0; k < kSahThreads / 32; k++) {
                const int x = wl[k], y = wr[k];
                wl[k] = tl; wr[k] = tr;
                tl += x; tr += y;
            }
            base[0] = begin + atomicAdd(&g.cur_l, tl);
            base[1] = begin + nl + atomicAdd(&g.cur_r, tr);
        }
        __syncthreads();
        int pl = base[0] + wl[warp], pr = base[1] + wr[warp];
        const unsigned lt = (1u << lane) - 1u;
        int cmin[2][3], cmax[2][3];
#pragma unroll
        for (int s = 0; s < 2; s++)
#pragma unroll
            for (int k = 0; k < 3; k++) { cmin[s][k] = 0x7FFFFFFF; cmax[s][k] = (int)0x80000000; }
#pragma unroll
        for (int r = 0; r < kPer; r++) {
            if (in[r]) {
                const int o = left[r] ? pl + __popc(ml[r] & lt) : pr + __popc(mr[r] & lt);
                if (o >= (left[r] ? begin : begin + nl) && o < (left[r] ? begin + nl : begin + count)) {
                    lo2[o] = a[r];
                    hi2[o] = b[r];
                } else {
                    atomicExch(bad, 11);
                }
                const int e[3] = {ord_of(sah_centre(a[r].x, b[r].x)), ord_of(sah_centre(a[r].y, b[r].y)),
                                  ord_of(sah_centre(a[r].z, b[r].z))};
#pragma unroll
                for (int k = 0; k < 3; k++) {
                    if (left[r]) { cmin[0][k] = min(cmin[0][k], e[k]); cmax[0][k] = max(cmax[0][k], e[k]); }
                    else { cmin[1][k] = min(cmin[1][k], e[k]); cmax[1][k] = max(cmax[1][k], e[k]); }
                }
                if (g.refs & (left[r] ? 1 : 2)) {       // a child that is this one cluster
                    int4 *ref = &nodes[g.node].r;
                    if (left[r]) ref->x = __float_as_int(a[r].w);
                    else ref->y = __float_as_int(a[r].w);
                }
            }
            pl += __popc(ml[r]);
            pr += __popc(mr[r]);
        }
        const int child[2] = {g.child_l, g.child_r};
#pragma unroll
        for (int s = 0; s < 2; s++)
            if (child[s] >= 0) {
#pragma unroll
                for (int k = 0; k < 3; k++) {
                    const int x = warp_min(cmin[s][k]), y = warp_max(cmax[s][k]);
                    if (lane == 0) { atomicMin(&cb[6 * s + k], x); atomicMax(&cb[6 * s + 3 + k], y); }
                }
            }
        __syncthreads();
        if (threadIdx.x < 12) {
            const int s = threadIdx.x / 6, k = threadIdx.x % 6;
            if (child[s] >= 0) {
                if (k < 3) atomicMin(&next[child[s]].clo[k], cb[threadIdx.x]);
                else atomicMax(&next[child[s]].chi[k - 3], cb[threadIdx.x]);
            }
        }
        __syncthreads();
    }
}

// Small segments, one warp each (taken from a counter): the clusters' boxes are loaded into
// shared memory once, and the warp splits index ranges depth-first, the larger side pushed
// (at most 8 pending), with the same bins and costs as the large segments; up to kSahSweep
// clusters it tries every plane instead, a lane each, which takes a tenth of the instructions
// of filling and scanning the bins (0.67 -> 0.38 ms at 265k clusters).  A segment of n clusters
// reserves its n - 1 nodes with one atomic.
constexpr int kSmallWarps = 4;
struct SahSmallWarp {
    float4 lo[kSahSmall], hi[kSahSmall];
    int bins[kSahSlotInts];
    uint8_t idx[kSahSmall];
    int4 stack[12];                      // (first, count, node, level)
};

__global__ void __launch_bounds__(kSmallWarps * 32) k_sah_small(SahState *st, int max_small, const int4 *small,
                                                                const float4 *lo0, const float4 *hi0, const float4 *lo1,
                                                                const float4 *hi1, BvhNode *nodes, int n_nodes,
                                                                int *node_count, int *bad) {
    extern __shared__ unsigned char sm_small[];
    SahSmallWarp &S = reinterpret_cast<SahSmallWarp *>(sm_small)[threadIdx.x >> 5];
    const unsigned lane = threadIdx.x & 31, lt = (1u << lane) - 1u;
    const int n = min(st->n_small, max_small);
    while (true) {
        int t = 0;
        if (lane == 0) t = atomicAdd(&st->small_next, 1);
        t = __shfl_sync(0xffffffffu, t, 0);
        if (t >= n) return;
        const int4 seg = small[t];
        const int begin = seg.x, count = seg.y;
        // the level a segment was made at tells which copy of the clusters holds it
        const float4 *lo = (seg.w & 1) ? lo1 : lo0, *hi = (seg.w & 1) ? hi1 : hi0;
        for (int k = (int)lane; k < count; k += 32) {
            S.lo[k] = lo[begin + k];
            S.hi[k] = hi[begin + k];
            S.idx[k] = (uint8_t)k;
        }
        int fresh = 0;                   // the next of the reserved nodes
        if (lane == 0 && count > 2) fresh = atomicAdd(node_count, count - 2);
        fresh = __shfl_sync(0xffffffffu, fresh, 0);
        if (fresh + max(count - 2, 0) > n_nodes || seg.z < 0 || seg.z >= n_nodes) {
            if (lane == 0) atomicExch(bad, 10);
            return;
        }
        __syncwarp();
        int first = 0, cnt = count, node = seg.z, level = seg.w, sp = 0;
        while (true) {
            int nl = 1;
            float bl[2][3], bh[2][3];
            if (cnt == 2) {
#pragma unroll
                for (int s = 0; s < 2; s++) {
                    const float4 a = S.lo[S.idx[first + s]], b = S.hi[S.idx[first + s]];
                    bl[s][0] = a.x; bl[s][1] = a.y; bl[s][2] = a.z;
                    bh[s][0] = b.x; bh[s][1] = b.y; bh[s][2] = b.z;
                }
            } else if (cnt <= kSahSweep) {
                // every plane of every axis: lane (axis, k) puts the clusters up to the k-th one's
                // centre (ties by position) on the left
                const int axis = (int)lane / cnt, i = (int)lane - axis * cnt;
                const bool mine = axis < 3;
                auto centre = [&](const float4 &a, const float4 &b, int ax) {
                    return ax == 0 ? sah_centre(a.x, b.x) : (ax == 1 ? sah_centre(a.y, b.y) : sah_centre(a.z, b.z));
                };
                const int own = S.idx[first + i];
                const float ci = centre(S.lo[own], S.hi[own], axis);
                float cost = INFINITY;
                int n = 0;
#pragma unroll
                for (int s = 0; s < 2; s++)
#pragma unroll
                    for (int q = 0; q < 3; q++) { bl[s][q] = INFINITY; bh[s][q] = -INFINITY; }
                for (int k = 0; k < cnt; k++) {
                    const int o = S.idx[first + k];
                    const float4 a = S.lo[o], b = S.hi[o];
                    const float ck = centre(a, b, axis);
                    if (ck < ci || (ck == ci && k <= i)) {
                        n++;
                        bl[0][0] = fminf(bl[0][0], a.x); bl[0][1] = fminf(bl[0][1], a.y); bl[0][2] = fminf(bl[0][2], a.z);
                        bh[0][0] = fmaxf(bh[0][0], b.x); bh[0][1] = fmaxf(bh[0][1], b.y); bh[0][2] = fmaxf(bh[0][2], b.z);
                    } else {
                        bl[1][0] = fminf(bl[1][0], a.x); bl[1][1] = fminf(bl[1][1], a.y); bl[1][2] = fminf(bl[1][2], a.z);
                        bh[1][0] = fmaxf(bh[1][0], b.x); bh[1][1] = fmaxf(bh[1][1], b.y); bh[1][2] = fmaxf(bh[1][2], b.z);
                    }
                }
                if (mine && n > 0 && n < cnt)
                    cost = half_area(make_float4(bl[0][0], bl[0][1], bl[0][2], 0.f), make_float4(bh[0][0], bh[0][1], bh[0][2], 0.f)) * (float)n +
                           half_area(make_float4(bl[1][0], bl[1][1], bl[1][2], 0.f), make_float4(bh[1][0], bh[1][1], bh[1][2], 0.f)) * (float)(cnt - n);
                if (!(cost < INFINITY)) cost = INFINITY;
                const int low = __reduce_min_sync(0xffffffffu, ord_of(cost));
                const unsigned at = __ballot_sync(0xffffffffu, mine && cost < INFINITY && ord_of(cost) == low);
                if (at == 0u || level >= kSahMaxLevel) {
                    // no plane: by position, both sides with the box of all
                    nl = cnt / 2;
#pragma unroll
                    for (int q = 0; q < 3; q++) {
                        bl[0][q] = bl[1][q] = float_of(warp_min(ord_of(fminf(bl[0][q], bl[1][q]))));
                        bh[0][q] = bh[1][q] = float_of(warp_max(ord_of(fmaxf(bh[0][q], bh[1][q]))));
                    }
                } else {
                    const int win = __ffs(at) - 1, wa = win / cnt, wi = win - wa * cnt;
                    nl = __shfl_sync(0xffffffffu, n, win);
#pragma unroll
                    for (int s = 0; s < 2; s++)
#pragma unroll
                        for (int q = 0; q < 3; q++) {
                            bl[s][q] = __shfl_sync(0xffffffffu, bl[s][q], win);
                            bh[s][q] = __shfl_sync(0xffffffffu, bh[s][q], win);
                        }
                    const float cw = __shfl_sync(0xffffffffu, ci, win);
                    uint8_t v = 0;
                    bool left = false;
                    if ((int)lane < cnt) {
                        v = S.idx[first + (int)lane];
                        const float ck = centre(S.lo[v], S.hi[v], wa);
                        left = ck < cw || (ck == cw && (int)lane <= wi);
                    }
                    const unsigned m = __ballot_sync(0xffffffffu, left), all = (1u << cnt) - 1u;
                    __syncwarp();
                    if ((int)lane < cnt) {
                        const int o = left ? __popc(m & lt) : nl + __popc(~m & all & lt);
                        if (o < cnt) S.idx[first + o] = v;
                        else atomicExch(bad, 11);
                    }
                }
                __syncwarp();
            } else {
                // the centroids' bounds, then the bins
                int l[3] = {0x7FFFFFFF, 0x7FFFFFFF, 0x7FFFFFFF}, h[3] = {(int)0x80000000, (int)0x80000000, (int)0x80000000};
                for (int k = (int)lane; k < cnt; k += 32) {
                    const float4 a = S.lo[S.idx[first + k]], b = S.hi[S.idx[first + k]];
                    const int e[3] = {ord_of(sah_centre(a.x, b.x)), ord_of(sah_centre(a.y, b.y)), ord_of(sah_centre(a.z, b.z))};
#pragma unroll
                    for (int q = 0; q < 3; q++) { l[q] = min(l[q], e[q]); h[q] = max(h[q], e[q]); }
                }
                float cl[3], ext[3];
#pragma unroll
                for (int q = 0; q < 3; q++) {
                    cl[q] = float_of(warp_min(l[q]));
                    ext[q] = __fsub_rn(float_of(warp_max(h[q])), cl[q]);
                }
                sah_bins_clear(S.bins, (int)lane, 32);
                __syncwarp();
                for (int k = (int)lane; k < cnt; k += 32) {
                    const float4 a = S.lo[S.idx[first + k]], b = S.hi[S.idx[first + k]];
                    const int bin[3] = {sah_bin(sah_centre(a.x, b.x), cl[0], ext[0]), sah_bin(sah_centre(a.y, b.y), cl[1], ext[1]),
                                        sah_bin(sah_centre(a.z, b.z), cl[2], ext[2])};
                    sah_bins_add(S.bins, bin, a, b);
                }
                __syncwarp();
                SahPlane p = sah_select(S.bins, lane);
                if (level >= kSahMaxLevel || p.nl <= 0 || p.nl >= cnt) p.axis = -1;
                if (p.axis < 0) {
                    p.nl = cnt / 2;
#pragma unroll
                    for (int q = 0; q < 3; q++) {
                        const int *b = S.bins + (lane & 15u);
                        p.lo[0][q] = p.lo[1][q] = float_of(warp_min(b[(1 + q) * kSahBins]));
                        p.hi[0][q] = p.hi[1][q] = float_of(warp_max(b[(4 + q) * kSahBins]));
                    }
                } else {
                    // stable partition of the index range (all of it read before any is written)
                    uint8_t v[kSahSmall / 32];
                    unsigned m[kSahSmall / 32];
                    const float pcl = p.axis == 0 ? cl[0] : (p.axis == 1 ? cl[1] : cl[2]);
                    const float pex = p.axis == 0 ? ext[0] : (p.axis == 1 ? ext[1] : ext[2]);
#pragma unroll
                    for (int r = 0; r < kSahSmall / 32; r++) {
                        m[r] = 0u;
                        v[r] = 0;
                        if (r * 32 < cnt) {
                            const int k = r * 32 + (int)lane;
                            bool left = false;
                            if (k < cnt) {
                                v[r] = S.idx[first + k];
                                const float4 a = S.lo[v[r]], b = S.hi[v[r]];
                                const float c = p.axis == 0 ? sah_centre(a.x, b.x) : (p.axis == 1 ? sah_centre(a.y, b.y) : sah_centre(a.z, b.z));
                                left = sah_bin(c, pcl, pex) <= p.bin;
                            }
                            m[r] = __ballot_sync(0xffffffffu, left);
                        }
                    }
                    __syncwarp();
                    int ol = first, orr = first + p.nl;
#pragma unroll
                    for (int r = 0; r < kSahSmall / 32; r++) {
                        if (r * 32 < cnt) {
                            const int k = r * 32 + (int)lane;
                            const unsigned in = cnt - r * 32 >= 32 ? 0xffffffffu : (1u << (cnt - r * 32)) - 1u;
                            if (k < cnt) {
                                const int o = ((m[r] >> lane) & 1u) ? ol + __popc(m[r] & lt) : orr + __popc(~m[r] & in & lt);
                                if (o < first + cnt) S.idx[o] = v[r];
                                else atomicExch(bad, 11);
                            }
                            ol += __popc(m[r]);
                            orr += __popc(~m[r] & in);
                        }
                    }
                }
                nl = p.nl;
#pragma unroll
                for (int s = 0; s < 2; s++)
#pragma unroll
                    for (int q = 0; q < 3; q++) { bl[s][q] = p.lo[s][q]; bh[s][q] = p.hi[s][q]; }
                __syncwarp();
            }
            const int nr = cnt - nl;
            int ref[2];
            ref[0] = nl == 1 ? __float_as_int(S.lo[S.idx[first]].w) : fresh++;
            ref[1] = nr == 1 ? __float_as_int(S.lo[S.idx[first + nl]].w) : fresh++;
            if (lane == 0)
                nodes[node] = make_node(make_float4(bl[0][0], bl[0][1], bl[0][2], 0.f), make_float4(bh[0][0], bh[0][1], bh[0][2], 0.f),
                                        ref[0], make_float4(bl[1][0], bl[1][1], bl[1][2], 0.f),
                                        make_float4(bh[1][0], bh[1][1], bh[1][2], 0.f), ref[1]);
            level++;
            if (nl > 1 && nr > 1) {
                const bool big_left = nl >= nr;
                if (lane == 0)
                    S.stack[sp] = big_left ? make_int4(first, nl, ref[0], level) : make_int4(first + nl, nr, ref[1], level);
                sp++;
                if (big_left) { first += nl; cnt = nr; node = ref[1]; }
                else { cnt = nl; node = ref[0]; }
            } else if (nl > 1) {
                cnt = nl; node = ref[0];
            } else if (nr > 1) {
                first += nl; cnt = nr; node = ref[1];
            } else {
                if (sp == 0) break;
                __syncwarp();
                const int4 e = S.stack[--sp];
                first = e.x; cnt = e.y; node = e.z; level = e.w;
            }
            __syncwarp();
        }
        __syncwarp();
    }
}


// ---------------------------------------------------------------------------
// Collapse of the binary tree into 4-wide nodes, top-down one level per launch:
// a 4-wide node starts from the two children of its binary node and opens its
// largest-area internal child until it holds four children (or only leaves).  The
// child boxes are stored as the binary tree holds them.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void bin_child(const BvhNode &nd, int c, float3 &lo, float3 &hi, int &ref) {
    if (c == 0) {
        lo = make_float3(nd.a.x, nd.b.x, nd.c.x); hi = make_float3(nd.a.y, nd.b.y, nd.c.y); ref = nd.r.x;
    } else {
        lo = make_float3(nd.a.z, nd.b.z, nd.c.z); hi = make_float3(nd.a.w, nd.b.w, nd.c.w); ref = nd.r.y;
    }
}

// frontier counters: n4[0] 4-wide nodes made, n4[1 + level] the frontier of each level
constexpr int kCollapseLevels = 200;
__global__ void k_collapse_root(const int *root, int2 *f, int *n4) {
    n4[0] = n4[1] = 1;
    f[0] = make_int2(0, *root);
}

__global__ void __launch_bounds__(128) k_collapse(const BvhNode *nodes, int n_bin, const int2 *fin, const int *n_in, Bvh4Node *out4,
                                                  int max4, int *n4, int2 *fout, int *n_out, int *bad) {
  const int n = *n_in;
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < n; t += gridDim.x * blockDim.x) {
    int w4 = fin[t].x, b = fin[t].y;
    if (b < 0 || b >= n_bin || w4 < 0 || w4 >= max4) { atomicExch(bad, 5); return; }
    float3 lo[4], hi[4];
    int ref[4], cnt = 2;
    BvhNode nd = nodes[b];
    bin_child(nd, 0, lo[0], hi[0], ref[0]);
    bin_child(nd, 1, lo[1], hi[1], ref[1]);
    while (cnt < 4) {
        int best = -1;
        float ba = -1.f;
        for (int e = 0; e < cnt; e++) {
            if (ref[e] < 0) continue;
            float dx = hi[e].x - lo[e].x, dy = hi[e].y - lo[e].y, dz = hi[e].z - lo[e].z;
            float a = dx * dy + dy * dz + dz * dx;
            if (a > ba) { ba = a; best = e; }
        }
        if (best < 0) break;
        if (ref[best] >= n_bin) { atomicExch(bad, 5); return; }
        BvhNode c = nodes[ref[best]];
        bin_child(c, 0, lo[best], hi[best], ref[best]);
        bin_child(c, 1, lo[cnt], hi[cnt], ref[cnt]);
        cnt++;
    }
    int nint = 0;
    for (int e = 0; e < cnt; e++) nint += ref[e] >= 0;
    int base = nint ? atomicAdd(n4, nint) : 0;
    if (base + nint > max4) { atomicExch(bad, 6); return; }
    int fo = nint ? atomicAdd(n_out, nint) : 0;
    if (fo + nint > max4) { atomicExch(bad, 6); return; }
    float L[3][4], Hh[3][4];
    int R[4];
    int k = 0;
    for (int e = 0; e < 4; e++) {
        if (e < cnt) {
            L[0][e] = lo[e].x;
            L[1][e] = lo[e].y;
            L[2][e] = lo[e].z;
            Hh[0][e] = hi[e].x;
            Hh[1][e] = hi[e].y;
            Hh[2][e] = hi[e].z;
            if (ref[e] >= 0) {
                R[e] = base + k;
                fout[fo + k] = make_int2(base + k, ref[e]);
                k++;
            } else {
                R[e] = ref[e];
            }
        } else {
            L[0][e] = L[1][e] = L[2][e] = 0.f;
            Hh[0][e] = Hh[1][e] = Hh[2][e] = 0.f;
            R[e] = kEmptyChild;
        }
    }
    Bvh4Node o;
    o.lox = make_float4(L[0][0], L[0][1], L[0][2], L[0][3]);
    o.hix = make_float4(Hh[0][0], Hh[0][1], Hh[0][2], Hh[0][3]);
    o.loy = make_float4(L[1][0], L[1][1], L[1][2], L[1][3]);
    o.hiy = make_float4(Hh[1][0], Hh[1][1], Hh[1][2], Hh[1][3]);
    o.loz = make_float4(L[2][0], L[2][1], L[2][2], L[2][3]);
    o.hiz = make_float4(Hh[2][0], Hh[2][1], Hh[2][2], Hh[2][3]);
    o.ref = make_int4(R[0], R[1], R[2], R[3]);
    o.pad = make_int4(0, 0, 0, 0);
    out4[w4] = o;
  }
}

// what the host needs to know of the finished tree
struct TreeSummary {
    int bad, depth, root;
    float lo[3], hi[3];                  // the root's box
};
__global__ void k_summary(const int *ibuf, const int *root, const BvhNode *nodes, int n_nodes, TreeSummary *o) {
    o->bad = ibuf[6];
    o->depth = ibuf[7];
    o->root = *root;
    if (*root >= 0 && *root < n_nodes) {
        const BvhNode nd = nodes[*root];
        o->lo[0] = fminf(nd.a.x, nd.a.z); o->lo[1] = fminf(nd.b.x, nd.b.z); o->lo[2] = fminf(nd.c.x, nd.c.z);
        o->hi[0] = fmaxf(nd.a.y, nd.a.w); o->hi[1] = fmaxf(nd.b.y, nd.b.w); o->hi[2] = fmaxf(nd.c.y, nd.c.w);
    }
}

// ---------------------------------------------------------------------------
// device exclusive scan (int) and stable LSD radix sort (64-bit keys, 32-bit values)
// ---------------------------------------------------------------------------
constexpr int kScanThreads = 256, kScanItems = 8, kScanTile = kScanThreads * kScanItems;

// exclusive prefix of v over the 256 threads of the block; *total = the block's sum
__device__ __forceinline__ int block_exclusive_scan(int v, int *warp_sums, int &total) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    int incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
    }
    if (lane == 31) warp_sums[w] = incl;
    __syncthreads();
    int wpre = 0, tot = 0;
#pragma unroll
    for (int k = 0; k < kScanThreads / 32; k++) {
        const int s = warp_sums[k];
        if (k < w) wpre += s;
        tot += s;
    }
    __syncthreads();
    total = tot;
    return wpre + incl - v;
}

// tile-local exclusive prefix of in[0..n) into out, and each tile's sum into sums
__global__ void __launch_bounds__(kScanThreads) k_scan_tiles(const int *in, int *out, int n, int *sums) {
    __shared__ int ws[kScanThreads / 32];
    const long long base = (long long)blockIdx.x * kScanTile + (long long)threadIdx.x * kScanItems;
    int v[kScanItems], s = 0;
#pragma unroll
    for (int k = 0; k < kScanItems; k++) {
        v[k] = base + k < n ? in[base + k] : 0;
        s += v[k];
    }
    int tot;
    int pre = block_exclusive_scan(s, ws, tot);
#pragma unroll
    for (int k = 0; k < kScanItems; k++) {
        if (base + k < n) out[base + k] = pre;
        pre += v[k];
    }
    if (threadIdx.x == 0) sums[blockIdx.x] = tot;
}

// exclusive prefix of sums[0..nb) in place, one block (each thread a consecutive chunk)
__global__ void __launch_bounds__(kScanThreads) k_scan_sums(int *sums, int nb) {
    __shared__ int ws[kScanThreads / 32];
    const int chunk = (nb + kScanThreads - 1) / kScanThreads;
    const int b0 = threadIdx.x * chunk;
    int s = 0;
    for (int k = 0; k < chunk; k++)
        if (b0 + k < nb) s += sums[b0 + k];
    int tot;
    int pre = block_exclusive_scan(s, ws, tot);
    for (int k = 0; k < chunk; k++)
        if (b0 + k < nb) {
            const int v = sums[b0 + k];
            sums[b0 + k] = pre;
            pre += v;
        }
}

__global__ void k_scan_add(int *out, int n, const int *sums) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] += sums[i / kScanTile];
}

// out[i] = in[0] + ... + in[i-1]; sums holds ceil(n / 2048) ints
void device_exclusive_scan(const int *in, int *out, int n, int *sums, cudaStream_t st) {
    if (n <= 0) return;
    const int nb = (n + kScanTile - 1) / kScanTile;
    k_scan_tiles<<<nb, kScanThreads, 0, st>>>(in, out, n, sums);
    k_scan_sums<<<1, kScanThreads, 0, st>>>(sums, nb);
    k_scan_add<<<(n + 255) / 256, 256, 0, st>>>(out, n, sums);
}

constexpr int kSortThreads = 256, kSortRounds = 8, kSortTile = kSortThreads * kSortRounds, kSortBins = 256;

// per block of 2048 keys: the count of each 8-bit digit at `shift`, digit-major
__global__ void __launch_bounds__(kSortThreads) k_rs_hist(const unsigned long long *keys, int n, int shift, int *hist,
                                                          int nblocks) {
    __shared__ int h[kSortBins];
    h[threadIdx.x] = 0;
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kSortRounds; r++) {
        const long long idx = (long long)blockIdx.x * kSortTile + r * kSortThreads + threadIdx.x;
        if (idx < n) atomicAdd(&h[(int)((keys[idx] >> shift) & 255ull)], 1);
    }
    __syncthreads();
    hist[threadIdx.x * nblocks + blockIdx.x] = h[threadIdx.x];
}

// Stable scatter of a block's 2048 keys by their digit: offs[d * nblocks + b] is where
// digit d of block b starts (exclusive scan of the histograms).  The block takes its keys
// in 8 rounds of 256 in index order; within a round a key's place among equal digits is
// its rank in its warp (lanes with the same digit, __match_any_sync) plus the counts of
// the lower warps, and the digit's running offset carries across rounds.
__global__ void __launch_bounds__(kSortThreads) k_rs_scatter(const unsigned long long *keys, const uint32_t *vals,
                                                             unsigned long long *keys_out, uint32_t *vals_out, int n,
                                                             int shift, const int *offs, int nblocks) {
    __shared__ int run[kSortBins];
    __shared__ int wcount[kSortThreads / 32][kSortBins];
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const unsigned lt = (1u << lane) - 1u;
    run[tid] = offs[tid * nblocks + blockIdx.x];
    for (int r = 0; r < kSortRounds; r++) {
        const long long idx = (long long)blockIdx.x * kSortTile + r * kSortThreads + tid;
        const bool valid = idx < n;
        const unsigned long long key = valid ? keys[idx] : 0ull;
        const uint32_t val = valid ? vals[idx] : 0u;
        const int d = valid ? (int)((key >> shift) & 255ull) : kSortBins;
#pragma unroll
        for (int k = 0; k < kSortBins / 32; k++) wcount[w][lane + 32 * k] = 0;
        __syncwarp();
        const unsigned peers = __match_any_sync(0xffffffffu, d);
        const int rank = __popc(peers & lt);
        if (valid && lane == __ffs(peers) - 1) wcount[w][d] = __popc(peers);
        __syncthreads();
        // per digit (thread tid = digit tid): exclusive prefix of the warps' counts
        int acc = 0;
#pragma unroll
        for (int k = 0; k < kSortThreads / 32; k++) {
            const int c = wcount[k][tid];
            wcount[k][tid] = acc;
            acc += c;
        }
        __syncthreads();
        if (valid) {
            const int pos = run[d] + wcount[w][d] + rank;
            keys_out[pos] = key;
            vals_out[pos] = val;
        }
        __syncthreads();
        run[tid] += acc;
        __syncthreads();
    }
}

// Stable sort of (keys, vals) by bits [from, to) of the keys (a multiple of 16 of them: an even
// number of 8-bit passes); the result ends in (keys, vals), (keys2, vals2) and hist are
// scratch (hist: 256 * ceil(n / 2048) ints, sums: ceil(256 * ceil(n / 2048) / 2048) ints).
void device_radix_sort_pairs(unsigned long long *keys, uint32_t *vals, unsigned long long *keys2, uint32_t *vals2,
                             int n, int *hist, int *sums, cudaStream_t st, int from = 0, int to = 64) {
    if (n <= 1) return;
    const int nb = (n + kSortTile - 1) / kSortTile;
    unsigned long long *ki = keys, *ko = keys2;
    uint32_t *vi = vals, *vo = vals2;
    for (int shift = from; shift < to; shift += 8) {
        k_rs_hist<<<nb, kSortThreads, 0, st>>>(ki, n, shift, hist, nb);
        device_exclusive_scan(hist, hist, kSortBins * nb, sums, st);
        k_rs_scatter<<<nb, kSortThreads, 0, st>>>(ki, vi, ko, vo, n, shift, hist, nb);
        unsigned long long *tk = ki; ki = ko; ko = tk;
        uint32_t *tv = vi; vi = vo; vo = tv;
    }
    // an even number of passes: the sorted data are back in (keys, vals)
}

}  // namespace

size_t sort_pairs_scratch_ints(int n) {
    const size_t nbk = (size_t)(n + kSortTile - 1) / kSortTile;
    const size_t nh = (size_t)kSortBins * nbk;
    return nh + (nh + kScanTile - 1) / kScanTile + 1;
}

void sort_pairs_by_low_bits(unsigned long long *keys, uint32_t *vals, unsigned long long *keys2, uint32_t *vals2,
                            int n, int bits, int *scratch, cudaStream_t st) {
    const size_t nh = (size_t)kSortBins * ((n + kSortTile - 1) / kSortTile);
    device_radix_sort_pairs(keys, vals, keys2, vals2, n, scratch, scratch + nh, st, 0, bits);
}

static inline unsigned blocks_for(size_t n, int b) { return (unsigned)((n + b - 1) / b); }

namespace {
// One block of scratch, handed out in 256-byte aligned pieces (sized first, then taken).
struct Arena {
    char *base = nullptr;
    size_t used = 0;
    template <class T> T *take(size_t n) {
        T *p = base ? reinterpret_cast<T *>(base + used) : nullptr;
        used += (n * sizeof(T) + 255) & ~(size_t)255;
        return p;
    }
};

struct BuildScratch {
    float4 *cen;
    int *ibuf;                           // [0..5] centroid bounds, [6] bad, [7] depth, [8] large count, [9..14] small
                                         // bounds, [15] nodes made
    int *root;
    unsigned long long *keys, *keys2;
    uint32_t *vals, *vals2;
    int *hist, *sums;                    // radix sort and scan
    int *pnode, *pleaf, *arr;
    TreeSummary *summary;
    SahState *state;
    // Karras
    int4 *child;
    float4 *blo, *bhi;
    // PLOC and SAH
    float4 *clo[2], *chi[2];
    int *nn, *keep, *pos;
    SahSeg *segs[2];
    int *bins[2];
    int2 *items[2];
    int4 *small;
    int max_segs, max_items, max_small;
    // collapse
    Bvh4Node *wide;
    int2 *front[2];
    int *n4;

    void lay_out(Arena &A, int n, bool ploc) {
        const size_t nn1 = (size_t)std::max(n - 1, 1);
        const size_t nbk = (size_t)(n + kSortTile - 1) / kSortTile, nh = (size_t)kSortBins * nbk;
        cen = A.take<float4>(n);
        ibuf = A.take<int>(16);
        root = A.take<int>(1);
        keys = A.take<unsigned long long>(n);
        keys2 = A.take<unsigned long long>(n);
        vals = A.take<uint32_t>(n);
        vals2 = A.take<uint32_t>(n);
        hist = A.take<int>(nh);
        sums = A.take<int>(std::max((nh + kScanTile - 1) / kScanTile, (size_t)(n + kScanTile - 1) / kScanTile) + 1);
        pnode = A.take<int>(nn1);
        pleaf = A.take<int>(n);
        arr = A.take<int>(nn1);
        summary = A.take<TreeSummary>(1);
        state = A.take<SahState>(1);
        max_segs = n / (kSahSmall + 1) + 2;
        max_items = n / kSahChunk + max_segs + 2;
        max_small = n / 2 + 2;
        if (ploc) {
            for (int k = 0; k < 2; k++) {
                clo[k] = A.take<float4>(n);
                chi[k] = A.take<float4>(n);
                segs[k] = A.take<SahSeg>(max_segs);
                bins[k] = A.take<int>((size_t)max_segs * kSahSlotInts);
                items[k] = A.take<int2>(max_items);
            }
            nn = A.take<int>(n);
            keep = A.take<int>(n);
            pos = A.take<int>(n);
            small = A.take<int4>(max_small);
        } else {
            child = A.take<int4>(nn1);
            blo = A.take<float4>(2 * (size_t)n);
            bhi = A.take<float4>(2 * (size_t)n);
        }
        wide = A.take<Bvh4Node>(nn1);
        for (int k = 0; k < 2; k++) front[k] = A.take<int2>(nn1);
        n4 = A.take<int>(kCollapseLevels + 2);
    }
};

// levels [from, from + count) of the large segments
void sah_levels(const BuildScratch &b, DofScene *s, int m, int from, int count, int sms, cudaStream_t st) {
    for (int l = from; l < from + count; l++) {
        const int p = l & 1;
        k_sah_bin<<<4 * sms, kSahThreads, 0, st>>>(b.state, p, b.segs[p], b.items[p], b.clo[p], b.chi[p], b.bins[p]);
        k_sah_split<<<sms, 128, 0, st>>>(b.state, p, b.segs[p], b.bins[p], b.segs[p ^ 1], b.bins[p ^ 1], b.items[p ^ 1],
                                         b.max_segs, b.max_items, b.small, b.max_small, s->nodes, m - 1, b.ibuf + 15,
                                         b.ibuf + 6);
        k_sah_part<<<4 * sms, kSahThreads, 0, st>>>(b.state, p, b.segs[p], b.items[p], b.clo[p], b.chi[p], b.clo[p ^ 1],
                                                    b.chi[p ^ 1], b.segs[p ^ 1], s->nodes, b.ibuf + 6);
    }
}

// The hierarchy over the m >= 2 sorted tree triangles: one PLOC round, then SAH.
int ploc_sah_build(const BuildScratch &b, DofScene *s, int m, int radius, int sms, cudaStream_t st) {
    const int B = 256;
    int rc = DOF_OK;
    auto ck = [&](cudaError_t e, const char *w) { if (rc == DOF_OK && e != cudaSuccess) rc = dof_cuda_check(e, w); };
    // the clusters are compacted into copy 0 from copy 1
    k_ploc_init<<<blocks_for(m, B), B, 0, st>>>(s->tris, m, b.clo[1], b.chi[1]);
    radius = std::min(std::max(radius, 1), kNnMaxRadius);
    k_ploc_nn<<<blocks_for(m, kNnThreads), kNnThreads, (kNnThreads + 2 * radius) * 2 * sizeof(float4), st>>>(
        m, radius, b.clo[1], b.chi[1], b.nn);
    k_ploc_merge<<<blocks_for(m, B), B, 0, st>>>(m, b.clo[1], b.chi[1], b.nn, b.keep, b.ibuf + 15, s->nodes, m - 1, b.ibuf + 6);
    device_exclusive_scan(b.keep, b.pos, m, b.sums, st);
    k_ploc_scatter<<<blocks_for(m, B), B, 0, st>>>(m, b.keep, b.pos, b.clo[1], b.chi[1], b.clo[0], b.chi[0]);
    k_sah_root<<<1, 32, 0, st>>>(b.state, b.pos, b.keep, m, b.clo[0], b.segs[0], b.bins[0], b.items[0], b.max_items, b.small,
                                 b.ibuf + 15, b.root, b.ibuf + 6);
    if (m > kSahSmall) {
        k_sah_root_bounds<<<2 * sms, kSahThreads, 0, st>>>(b.state, b.clo[0], b.chi[0], b.segs[0]);
        // as many levels as balanced halving of the clusters (at most m) and a few uneven planes
        // take, then more while segments are left
        int levels = 4;
        while ((m >> 1 >> (levels - 4)) > kSahSmall) levels++;
        sah_levels(b, s, m, 0, levels, sms, st);
        for (int from = levels;; from += 4) {
            int left[2] = {0, 0};
            ck(cudaMemcpyAsync(left, b.state->n_seg, sizeof(left), cudaMemcpyDeviceToHost, st), "bvh levels");
            ck(cudaStreamSynchronize(st), "bvh levels");
            if (rc != DOF_OK || left[from & 1] == 0) break;
            if (from > 100) return dof_set_error(DOF_ERR_DEVICE_CHECK, "BVH splits did not end");
            sah_levels(b, s, m, from, 4, sms, st);
        }
    }
    const int shm = kSmallWarps * (int)sizeof(SahSmallWarp);
    k_sah_small<<<(int)std::min<size_t>(blocks_for(b.max_small, kSmallWarps), 5 * (size_t)sms), kSmallWarps * 32, shm, st>>>(
        b.state, b.max_small, b.small, b.clo[0], b.chi[0], b.clo[1], b.chi[1], s->nodes, m - 1, b.ibuf + 15, b.ibuf + 6);
    ck(cudaGetLastError(), "bvh kernels");
    return rc;
}

// The first key bit that the clustering round's sort looks at.  Its cells (10, 15 or 21 bits per axis
// of the centroids' extent) are at most two of the scene's median triangles wide, so that the
// order inside a cell, the input's, does not matter.  With ten bits whatever the scene, a lawn beside
// one triangle 14 km away, its triangles shuffled, took 120 node visits per packet ray instead
// of 58; with all of them every upload pays for eight passes instead of four (300k triangles 1565
// -> 1672 us, six passes 1622).
int cluster_key_from(const DofScene *s, const int *bounds) {
    float e[kSceneSamples];
    if (s->n_samples == 0) return 0;
    for (int k = 0; k < s->n_samples; k++) e[k] = s->sample[k][3];
    std::nth_element(e, e + s->n_samples / 2, e + s->n_samples);
    const float median = e[s->n_samples / 2];
    auto value = [](int o) {             // of an ordered int (ord_of)
        const int i = o >= 0 ? o : o ^ 0x7FFFFFFF;
        float f;
        memcpy(&f, &i, sizeof(f));
        return f;
    };
    float extent = 0.f;
    for (int k = 0; k < 3; k++) extent = std::max(extent, value(bounds[3 + k]) - value(bounds[k]));
    if (extent <= 2.f * 1024.f * median) return 32;
    if (extent <= 2.f * 32768.f * median) return 16;
    return 0;
}
}  // namespace

int launch_bvh_build(DofScene *s, const float *xyz, uint32_t n_verts, const uint32_t *idx, const uint32_t *mat, int builder, int ploc_radius, int rotations, cudaStream_t st) {
    const int n = (int)s->n_tris;
    const int B = 256, sms = s->ctx->sm_count;
    const bool ploc = builder == DOF_BVH_PLOC;
    const float share = ploc ? kLargeSah : kLargeLbvh;
    int rc = DOF_OK;
    auto ck = [&](cudaError_t e, const char *w) { if (rc == DOF_OK && e != cudaSuccess) rc = dof_cuda_check(e, w); };
    // all scratch in one stream-ordered block
    Arena arena;
    BuildScratch b{};
    b.lay_out(arena, n, ploc);
    float *d_xyz = arena.take<float>(3 * (size_t)n_verts);
    uint32_t *d_idx = arena.take<uint32_t>(3 * (size_t)n), *d_mat = mat ? arena.take<uint32_t>(n) : nullptr;
    rc = dof_scratch(s->ctx, arena.used, (void **)&arena.base, st, "bvh scratch");
    if (rc != DOF_OK) return rc;
    arena.used = 0;
    b.lay_out(arena, n, ploc);
    d_xyz = arena.take<float>(3 * (size_t)n_verts);
    d_idx = arena.take<uint32_t>(3 * (size_t)n);
    d_mat = mat ? arena.take<uint32_t>(n) : nullptr;
    ck(cudaMemcpyAsync(d_xyz, xyz, sizeof(float) * 3 * (size_t)n_verts, cudaMemcpyHostToDevice, st), "upload");
    ck(cudaMemcpyAsync(d_idx, idx, sizeof(uint32_t) * 3 * (size_t)n, cudaMemcpyHostToDevice, st), "upload");
    if (mat) ck(cudaMemcpyAsync(d_mat, mat, sizeof(uint32_t) * (size_t)n, cudaMemcpyHostToDevice, st), "upload");
    int hbuf[16];
    int n_small = n, n_big = 0;
    {
        const int lo_i = 0x7FFFFFFF, hi_i = (int)0x80000000;
        const int init[16] = {lo_i, lo_i, lo_i, hi_i, hi_i, hi_i, 0, 0, 0, lo_i, lo_i, lo_i, hi_i, hi_i, hi_i, 0};
        ck(cudaMemcpyAsync(b.ibuf, init, sizeof(init), cudaMemcpyHostToDevice, st), "bvh init");
        ck(cudaMemsetAsync(b.state, 0, sizeof(SahState), st), "bvh init");
        const unsigned gb = std::min(blocks_for(n, B), (unsigned)(4 * sms));
        k_centroids<<<gb, B, 0, st>>>(d_xyz, n_verts, d_idx, (uint32_t)n, b.cen, b.ibuf, b.ibuf + 6);
        k_classify<<<gb, B, 0, st>>>(b.cen, (uint32_t)n, b.ibuf, share, b.ibuf + 8, b.ibuf + 9);
        ck(cudaMemcpyAsync(hbuf, b.ibuf, sizeof(hbuf), cudaMemcpyDeviceToHost, st), "bvh readback");
        ck(cudaStreamSynchronize(st), "bvh classify");
        if (rc != DOF_OK) goto done;
        // large triangles stay out of the tree (tested directly by every ray) when there
        // are few of them and at least one other triangle
        int separate = hbuf[8] > 0 && hbuf[8] <= kMaxLargeTris && hbuf[8] < n;
        n_big = separate ? hbuf[8] : 0;
        n_small = n - n_big;
        k_morton<<<blocks_for(n, B), B, 0, st>>>(b.cen, (uint32_t)n, separate ? b.ibuf + 9 : b.ibuf, b.ibuf, share, separate,
                                                 b.keys, b.vals);
        // the radix tree needs the whole key, the clustering round as much of it as tells neighbours apart
        device_radix_sort_pairs(b.keys, b.vals, b.keys2, b.vals2, n, b.hist, b.sums, st,
                                ploc ? cluster_key_from(s, hbuf + (separate ? 9 : 0)) : 0, 64);
        // sorted (key, triangle) pairs are in (keys, vals)
        k_sorted_tris<<<blocks_for(n, B), B, 0, st>>>(d_xyz, d_idx, d_mat, (uint32_t)n, n_verts, b.vals, s->tris);
        const int m = n_small;
        int levels4 = 0, n_front[kCollapseLevels + 2];
        TreeSummary sum{};
        if (m >= 2) {
            ck(cudaMemsetAsync(s->nodes, 0xFF, sizeof(BvhNode) * (m - 1), st), "memset");
            if (ploc) {
                if (rc == DOF_OK) rc = ploc_sah_build(b, s, m, ploc_radius, sms, st);
                if (rc != DOF_OK) goto done;
            } else {
                ck(cudaMemsetAsync(b.arr, 0, sizeof(int) * (m - 1), st), "memset");
                ck(cudaMemsetAsync(b.root, 0, sizeof(int), st), "memset");
                k_karras<<<blocks_for(m - 1, B), B, 0, st>>>(b.keys, m, b.child, b.pnode, b.pleaf, b.ibuf + 6);
                k_refit<<<blocks_for(m, B), B, 0, st>>>(s->tris, m, b.child, b.pnode, b.pleaf, b.blo, b.bhi, b.arr, s->nodes,
                                                        b.ibuf + 6);
            }
            int *ref_leaf = reinterpret_cast<int *>(b.vals2);
            if (rotations > 0) {
                // the parents the passes walk up
                ck(cudaMemsetAsync(b.pnode, 0xFF, sizeof(int) * (m - 1), st), "memset");
                k_tree_refs<<<blocks_for(m - 1, B), B, 0, st>>>(s->nodes, m - 1, m, b.arr, ref_leaf, b.pnode, b.pleaf, b.ibuf + 6);
            }
            for (int pass = 0; pass < rotations; pass++) {
                ck(cudaMemsetAsync(b.arr, 0, sizeof(int) * (m - 1), st), "memset");
                k_rotate<<<blocks_for(m, B), B, 0, st>>>(m, s->nodes, b.pnode, b.pleaf, b.arr, b.ibuf + 6);
            }
            // the structure the packet tracer relies on (k_tree_refs), then the depth of
            // that structure; the sort's second buffers count the leaves' references
            ck(cudaMemsetAsync(b.arr, 0, sizeof(int) * (m - 1), st), "memset");
            ck(cudaMemsetAsync(b.vals2, 0, sizeof(int) * m, st), "memset");
            ck(cudaMemsetAsync(b.pnode, 0xFF, sizeof(int) * (m - 1), st), "memset");
            ck(cudaMemsetAsync(b.pleaf, 0xFF, sizeof(int) * m, st), "memset");
            k_tree_refs<<<blocks_for(m - 1, B), B, 0, st>>>(s->nodes, m - 1, m, b.arr, ref_leaf, b.pnode, b.pleaf, b.ibuf + 6);
            k_tree_counts<<<blocks_for(m, B), B, 0, st>>>(m - 1, m, b.root, b.arr, ref_leaf, b.ibuf + 6);
            k_depth<<<blocks_for(m, B), B, 0, st>>>(m, b.pnode, b.pleaf, b.ibuf + 7);
            // the 4-wide tree, level by level (a level past the deepest finds an empty frontier)
            ck(cudaMemsetAsync(b.n4, 0, sizeof(int) * (kCollapseLevels + 2), st), "memset");
            k_collapse_root<<<1, 1, 0, st>>>(b.root, b.front[0], b.n4);
            for (bool more = true; more && rc == DOF_OK;) {
                for (int k = 0; k < 16 && levels4 < kCollapseLevels; k++, levels4++)
                    k_collapse<<<2 * sms, 128, 0, st>>>(s->nodes, m - 1, b.front[levels4 & 1], b.n4 + 1 + levels4, b.wide, m - 1,
                                                       b.n4, b.front[(levels4 + 1) & 1], b.n4 + 2 + levels4, b.ibuf + 6);
                k_summary<<<1, 1, 0, st>>>(b.ibuf, b.root, s->nodes, m - 1, b.summary);
                ck(cudaMemcpyAsync(n_front, b.n4, sizeof(n_front), cudaMemcpyDeviceToHost, st), "bvh readback");
                ck(cudaMemcpyAsync(&sum, b.summary, sizeof(sum), cudaMemcpyDeviceToHost, st), "bvh readback");
                ck(cudaGetLastError(), "bvh kernels");
                ck(cudaStreamSynchronize(st), "bvh build");
                more = rc == DOF_OK && !sum.bad && n_front[1 + levels4] > 0 && levels4 < kCollapseLevels;
            }
        } else {
            ck(cudaMemcpyAsync(&sum.bad, b.ibuf + 6, sizeof(int), cudaMemcpyDeviceToHost, st), "bvh readback");
            ck(cudaGetLastError(), "bvh kernels");
            ck(cudaStreamSynchronize(st), "bvh build");
        }
        if (rc != DOF_OK) goto done;
        if (sum.bad == 1) { rc = dof_set_error(DOF_ERR_INVALID_ARG, "dof_scene_upload: vertex index out of range"); goto done; }
        if (sum.bad) { rc = dof_set_error(DOF_ERR_DEVICE_CHECK, "dof_scene_upload: BVH hierarchy check failed (%d)", sum.bad); goto done; }
        s->root = m >= 2 ? sum.root : ~0;
        s->depth = m >= 2 ? (uint32_t)sum.depth : 1;
        s->n_tree = (uint32_t)m;
        s->n_large = (uint32_t)n_big;
        s->n_nodes = m >= 2 ? (uint32_t)(m - 1) : 0;
        s->root4 = s->root;
        s->n_nodes4 = 0;
        s->depth4 = 0;
        if (s->depth > kTraversalStack) {
            rc = dof_set_error(DOF_ERR_DEVICE_CHECK, "BVH depth %u exceeds the traversal stack", s->depth);
            goto done;
        }
        if (m >= 2 && ploc) {
            // boxes whose areas overflow (or are no numbers) cannot be clustered by area
            const float dx = sum.hi[0] - sum.lo[0], dy = sum.hi[1] - sum.lo[1], dz = sum.hi[2] - sum.lo[2];
            if (!(dx * dy + dy * dz + dz * dx < INFINITY)) {
                rc = dof_set_error(DOF_ERR_DEVICE_CHECK, "dof_scene_upload: the triangles' bounds have no finite area");
                goto done;
            }
        }
        if (m >= 2) {
            if (n_front[1 + levels4] > 0) { rc = dof_set_error(DOF_ERR_DEVICE_CHECK, "BVH collapse did not terminate"); goto done; }
            while (s->depth4 < levels4 && n_front[1 + s->depth4] > 0) s->depth4++;
            s->n_nodes4 = n_front[0];
            s->nodes4_bytes = sizeof(Bvh4Node) * (size_t)s->n_nodes4;
            rc = dof_alloc(s->ctx, s->nodes4_bytes, (void **)&s->nodes4, &s->bytes);
            if (rc != DOF_OK) goto done;
            ck(cudaMemcpyAsync(s->nodes4, b.wide, s->nodes4_bytes, cudaMemcpyDeviceToDevice, st), "collapse copy");
            s->root4 = 0;
            // bounds of the tree's triangles
            for (int k = 0; k < 3; k++) { s->lo[k] = sum.lo[k]; s->hi[k] = sum.hi[k]; }
        }
    }
done:
    cudaFreeAsync(arena.base, st);
    return rc;
}
