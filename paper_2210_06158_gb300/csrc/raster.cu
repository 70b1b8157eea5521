// Object-order G-buffer producer (Section 3: the method shades a rasterised G-buffer).
//
// Visibility is resolved triangle by triangle instead of pixel by pixel: each triangle
// is set up once (its three edge planes through the lens centre give three half-planes
// of the image whose intersection holds every pixel centre whose primary ray can hit
// it), the pixels of that conservative region are enumerated, and each candidate pixel
// runs the same watertight ray/triangle test as the ray-cast producer.  The closest hit
// per pixel is the minimum of the 64-bit key (t bits, triangle id), which orders hits by
// distance and breaks exact ties on the smaller id, as the ray-cast producer does; a
// resolve pass shades it.  The two producers therefore give the same bits.
//
// Work distribution: triangles whose candidate box holds at most kSmallPx pixels are
// rasterised by the warp that set them up (the warp's 32 boxes are enumerated as one
// list, so a warp's lanes stay busy whatever the box sizes); larger ones are queued, and a
// warp takes each (or, above kChunkTiles, a stretch of its tiles): its lanes test 32 tiles of
// 8 x 8 pixels at once, then cover 32 surviving tiles at once, a bit per pixel; the pixels that
// are left form a list for the check against the closest hits, and those that pass a second
// one for the ray tests, so that each runs with all its lanes.
//
// Occlusion culling: the triangles are taken nearest first (sorted by a lower bound of their
// distance from the lens centre, its top 16 bits) in batches of growing size.  Before each
// batch, every pixel whose closest hit is nearer than the batch's least bound is marked done:
// no triangle from here on can win it.  A triangle whose candidate box holds only finished
// tiles is dropped whole, finished tiles and pixels of a queued triangle are dropped by their
// bits, and a candidate pixel skips the ray test when the bound is beyond the pixel's own
// closest hit.  Keys only decrease, so a stale read culls less, never wrongly; see near_bound
// for the margin.
//
// Bound: the workloads' candidate boxes hold 592 times the image's pixels at 1080p (496k
// triangles, tall blades in front of each other).  Enumerating them pixel by pixel took 6.4 of
// 8.4 ms; now 1.6 ms, of which the queued triangles 1.2 ms (the longest warps of each batch, and
// the tests of hits within a batch).  A farthest-hit pyramid over the tiles (4.7 ms) drops
// little: grass leaves gaps, and one far pixel keeps a tile open; the bits keep only that
// pixel.  Warps that take up to 1024 tiles set the time of a batch (4.3 ms); 64 tiles 1.9 ms, and
// with the lists 1.6 ms; 32 tiles 1.65 ms.  4, 6 and 8 batches: 2.0, 1.6 and 1.7 ms.
#include "geometry.cuh"

#include <algorithm>

namespace {

constexpr int kSmallPx = 64;         // candidate pixels above which a triangle is queued
// Tiles of a queued triangle that one warp takes at a time: one per 1024 triangles of the scene,
// between these.  In a scene of few triangles a few of them cover the image and have to be
// spread over the chip (256 x 144, 2.8k triangles: 159 us with 64 tiles, 59 us with 8); with
// many, claiming and looking up the pieces costs more than it spreads (1080p, 60k: 689 us with
// 64, 844 with 16, 1126 with 8; 640 x 360, 30k: 224, 190, 198).
constexpr int kChunkTiles = 64, kChunkTilesFew = 8;
constexpr int kRastThreads = 256;
constexpr int kBigThreads = 128;
constexpr int kTileShift = 3, kCoarseShift = 6;   // tiles of 8 x 8 and of 64 x 64 pixels
constexpr int kMaxFineTiles = 16;                 // boxes over more tiles are looked up in the coarse ones

// Edge functions of the image plane, scaled so that |a| + |b| = 1 (values in pixels)
// and oriented so that a pixel centre (x, y) can see the triangle only where
// a x + b y + c >= 0 for all three (after the safety margin added to c).
struct TriSetup {
    float e[9];                 // (a, b, c) per edge
    int i0, j0, i1, j1;         // candidate pixel box (inclusive)
};

// queued (large) triangle: setup and vertices
struct BigTri {
    float4 e0, e1, e2;          // (a, b, c, -) per edge
    int4 box;                   // i0, j0, i1, j1
    int k;                      // sorted triangle index
    float tn;                   // its distance bound (near_bound)
    int tiles;                  // 8 x 8 pixel tiles of the box
    int pad;
};

__device__ __forceinline__ float3 xyz(float4 v) { return make_float3(v.x, v.y, v.z); }
__device__ __forceinline__ float vlen(float3 v) { return sqrtf(dot(v, v)); }

__device__ __forceinline__ float edge_at(const float *e, float x, float y) { return fmaf(e[0], x, fmaf(e[1], y, e[2])); }

__device__ __forceinline__ bool edges_pass(const float *e, float x, float y) {
    return edge_at(e, x, y) >= 0.f && edge_at(e + 3, x, y) >= 0.f && edge_at(e + 6, x, y) >= 0.f;
}

// Conservative candidate region of one triangle.  Returns false when no pixel centre can
// see it.  Pixel (i, j) has its centre at (i + 1/2, j + 1/2); the primary ray direction
// of image point (x, y) is proportional to F + sx R - sy U with sx = (x + jx - W/2) / f,
// sy = (y + jy - H/2) / f (f the focal length in pixels).
//
// The ray with direction d hits the triangle at t > 0 exactly when d is a non-negative
// combination of the vertex offsets r_i = p_i - O, i.e. when e_k . d has the sign of
// D = det(r_0, r_1, r_2) for the three edge-plane normals e_k (e_0 = r_1 x r_2 ...).
// Each e_k . d is affine in (x, y) up to the positive factor of the normalisation, so
// the candidate region is an intersection of three half-planes; each is widened by
// half a pixel (far more than the rounding of either side), and its bounding box is
// found by clipping the image rectangle (its vertices are rectangle corners, line /
// rectangle-side crossings and line / line crossings).
__device__ bool tri_setup(const DevCam &cam, float4 v0, float4 v1, float4 v2, TriSetup &S) {
    const float3 p0 = xyz(v0), p1 = xyz(v1), p2 = xyz(v2);
    const float3 r0 = p0 - cam.O, r1 = p1 - cam.O, r2 = p2 - cam.O;
    const float3 g01 = p1 - p0, g12 = p2 - p1, g20 = p0 - p2;
    // a long vector times a short one: no cancellation for small, distant triangles
    const float3 e[3] = {cross(r1, g12), cross(r2, g20), cross(r0, g01)};
    const float D = -dot(g01, e[0]);     // (p0 - p1) . e0 = det(r0, r1, r2)
    const float Wf = (float)cam.W, Hf = (float)cam.H;
    const float xl = 0.5f, xh = Wf - 0.5f, yl = 0.5f, yh = Hf - 0.5f;
    // a plane through (or nearly through) the lens centre, an edge pointing at it, or a
    // degenerate triangle: the orientation is not reliable, so no edge is used and the
    // box is that of the projected vertices (the whole image if one is not in front)
    bool deg = !(fabsf(D) > 1e-5f * vlen(g01) * vlen(e[0]));
    deg = deg || !(vlen(e[0]) > 1e-5f * vlen(r1) * vlen(g12)) || !(vlen(e[1]) > 1e-5f * vlen(r2) * vlen(g20)) ||
          !(vlen(e[2]) > 1e-5f * vlen(r0) * vlen(g01));
    float xmin = INFINITY, xmax = -INFINITY, ymin = INFINITY, ymax = -INFINITY;
    if (deg) {
#pragma unroll
        for (int k = 0; k < 9; k++) S.e[k] = (k % 3 == 2) ? 1.f : 0.f;
        const float3 r[3] = {r0, r1, r2};
        bool front = true;
#pragma unroll
        for (int v = 0; v < 3; v++) {
            const float zc = dot(r[v], cam.F);
            if (!(zc > 0.f)) { front = false; continue; }
            const float x = cam.halfW - cam.jx + cam.Fpx * dot(r[v], cam.R) / zc;
            const float y = cam.halfH - cam.jy - cam.Fpx * dot(r[v], cam.U) / zc;
            xmin = fminf(xmin, x - 1.f); xmax = fmaxf(xmax, x + 1.f);
            ymin = fminf(ymin, y - 1.f); ymax = fmaxf(ymax, y + 1.f);
        }
        if (!front) { xmin = xl; xmax = xh; ymin = yl; ymax = yh; }
        if (!(xmin <= xmax) || !(ymin <= ymax)) return false;   // NaN vertices
    } else {
        const float s = D > 0.f ? 1.f : -1.f;
#pragma unroll
        for (int k = 0; k < 3; k++) {
            float a = dot(e[k], cam.R), b = -dot(e[k], cam.U);
            float c = dot(e[k], cam.F) * cam.Fpx + a * (cam.jx - cam.halfW) + b * (cam.jy - cam.halfH);
            if (c != c) return false;            // non-finite vertices: nothing to hit
            const float n = fabsf(a) + fabsf(b);
            const float sn = s / n, cn = c * sn;
            if (n > 0.f && fabsf(cn) < INFINITY) {
                a *= sn; b *= sn;
                c = cn + 0.5f + 1e-5f * (fabsf(cn) + Wf + Hf);
            } else {
                // the edge plane holds no image direction (or its line lies beyond float
                // range): one side of it sees the whole image, the other nothing
                c = (s * c >= 0.f) ? 1.f : -1.f;
                a = b = 0.f;
            }
            S.e[3 * k] = a; S.e[3 * k + 1] = b; S.e[3 * k + 2] = c;
        }
        // vertices of the clipped image rectangle; a candidate lying on a line is tested
        // only against the other lines, with a small tolerance
        const float tol = 1e-2f;
        auto inside_other = [&](float x, float y, int skip_a, int skip_b) {
            bool ok = true;
#pragma unroll
            for (int k = 0; k < 3; k++)
                if (k != skip_a && k != skip_b) ok = ok && edge_at(S.e + 3 * k, x, y) >= -tol;
            return ok;
        };
        auto add = [&](float x, float y) {
            xmin = fminf(xmin, x); xmax = fmaxf(xmax, x);
            ymin = fminf(ymin, y); ymax = fmaxf(ymax, y);
        };
        const float cx[2] = {xl, xh}, cy[2] = {yl, yh};
#pragma unroll
        for (int u = 0; u < 2; u++)
#pragma unroll
            for (int v = 0; v < 2; v++)
                if (inside_other(cx[u], cy[v], -1, -1)) add(cx[u], cy[v]);
#pragma unroll
        for (int k = 0; k < 3; k++) {
            const float a = S.e[3 * k], b = S.e[3 * k + 1], c = S.e[3 * k + 2];
            if (b != 0.f) {
#pragma unroll
                for (int u = 0; u < 2; u++) {
                    const float y = -(a * cx[u] + c) / b;
                    if (y >= yl - tol && y <= yh + tol && inside_other(cx[u], y, k, -1))
                        add(cx[u], fminf(fmaxf(y, yl), yh));
                }
            }
            if (a != 0.f) {
#pragma unroll
                for (int v = 0; v < 2; v++) {
                    const float x = -(b * cy[v] + c) / a;
                    if (x >= xl - tol && x <= xh + tol && inside_other(x, cy[v], k, -1))
                        add(fminf(fmaxf(x, xl), xh), cy[v]);
                }
            }
        }
#pragma unroll
        for (int k = 0; k < 3; k++) {
            const int l = (k + 1) % 3;
            const float ak = S.e[3 * k], bk = S.e[3 * k + 1], ck = S.e[3 * k + 2];
            const float al = S.e[3 * l], bl = S.e[3 * l + 1], cl = S.e[3 * l + 2];
            const float det = ak * bl - al * bk;
            if (det == 0.f) continue;
            const float x = (bk * cl - bl * ck) / det, y = (al * ck - ak * cl) / det;
            if (x >= xl - tol && x <= xh + tol && y >= yl - tol && y <= yh + tol && inside_other(x, y, k, l))
                add(fminf(fmaxf(x, xl), xh), fminf(fmaxf(y, yl), yh));
        }
        if (!(xmin <= xmax)) return false;
    }
    // pixel centres x = i + 1/2 in [xmin, xmax]
    S.i0 = max(0, (int)ceilf(fmaxf(xmin, 0.f) - 0.5f));
    S.i1 = min(cam.W - 1, (int)floorf(fminf(xmax, Wf) - 0.5f));
    S.j0 = max(0, (int)ceilf(fmaxf(ymin, 0.f) - 0.5f));
    S.j1 = min(cam.H - 1, (int)floorf(fminf(ymax, Hf) - 0.5f));
    return S.i0 <= S.i1 && S.j0 <= S.j1;
}

// q = idx / w, r = idx % w for idx < 2^22 through a float estimate and one correction
__device__ __forceinline__ void divmod(int idx, int w, float rw, int &q, int &r) {
    q = (int)(((float)idx + 0.5f) * rw);
    r = idx - q * w;
    if (r < 0) { q--; r += w; }
    else if (r >= w) { q++; r -= w; }
}

// the ray test of one candidate pixel, written to its closest-hit key
__device__ __forceinline__ void test_pixel(const DevCam &cam, unsigned long long *keys, int i, int j, float4 v0,
                                            float4 v1, float4 v2) {
    const float3 d = pixel_dir(cam, i + 0.5f, j + 0.5f);
    const Ray r = make_ray(cam.O, d);
    const float t = tri_hit(r, v0, v1, v2);
    if (t > 0.f && t < INFINITY) {
        const unsigned long long key =
            ((unsigned long long)__float_as_uint(t) << 32) | (unsigned long long)(uint32_t)__float_as_int(v0.w);
        atomicMin(&keys[(size_t)j * cam.W + i], key);
    }
}

// per batch: triangles queued whole; triangles cut into chunks (high word) and their chunks;
// the next piece of work
struct BigCounts {
    unsigned long long cut;
    uint32_t one, cursor;
};

// how triangles are cut: chunks of `tiles` tiles, more where a triangle would have over `most`
// chunks (so that a batch's work items fit 32 bits)
struct Cut {
    int tiles;
    uint32_t most;
    __device__ __forceinline__ uint32_t per_chunk(int n) const { return max((uint32_t)tiles, ((uint32_t)n + most - 1u) / most); }
};

struct SmallSlot {               // one triangle of a warp's list (112 bytes)
    float e[9];
    int i0, j0, bw;
    float rbw;
    float tn;                   // its distance bound (near_bound)
    int pad[2];
    float4 v0, v1, v2;
};

// Lower bound of the ray-test distance t of any primary ray to the triangle, for the
// occlusion test.  The directions are unit vectors, so t is the distance from the lens
// centre to the hit point, at least the distance to the triangle's bounding box, which
// is evaluated with every operation rounded down.  The test's t is a convex combination
// of the vertices' depths along the ray (barycentric weights), evaluated in FP32; the
// bound is shrunk by 2^-7 to stay below it.  A triangle with a vertex direction more than
// 60 degrees off the view axis (within 30 degrees of the lens plane) gets 0 and is never
// culled: near the lens plane those depths can cancel.
__device__ __forceinline__ float near_bound(const DevCam &cam, float4 v0, float4 v1, float4 v2) {
    const float4 v[3] = {v0, v1, v2};
#pragma unroll
    for (int k = 0; k < 3; k++) {
        const float3 r = make_float3(v[k].x - cam.O.x, v[k].y - cam.O.y, v[k].z - cam.O.z);
        if (!(dot(r, cam.F) >= 0.5f * sqrtf(dot(r, r)))) return 0.f;
    }
    auto gap = [](float o, float a, float b, float c) {
        const float lo = fminf(a, fminf(b, c)), hi = fmaxf(a, fmaxf(b, c));
        return fmaxf(fmaxf(__fsub_rd(lo, o), __fsub_rd(o, hi)), 0.f);
    };
    const float gx = gap(cam.O.x, v0.x, v1.x, v2.x), gy = gap(cam.O.y, v0.y, v1.y, v2.y);
    const float gz = gap(cam.O.z, v0.z, v1.z, v2.z);
    const float s = __fadd_rd(__fadd_rd(__fmul_rd(gx, gx), __fmul_rd(gy, gy)), __fmul_rd(gz, gz));
    const float d = __fmul_rd(__fsqrt_rd(s), 0.9921875f);
    return d >= 0.f ? d : 0.f;
}

// distance bits of a pixel's key: +inf while it has no hit
__device__ __forceinline__ uint32_t key_dist(unsigned long long key) { return min((uint32_t)(key >> 32), 0x7F800000u); }

// whether the pixel's closest hit so far is nearer than tn (from L2: the atomics update it there)
__device__ __forceinline__ bool occluded(const unsigned long long *keys, size_t q, float tn) {
    return tn > __uint_as_float(key_dist(__ldcg(&keys[q])));
}

// Which pixels are done (or outside the image): a bit each per 8 x 8 tile (row-major in the
// tile, tw x th tiles), and per 64 x 64 tile (tw2 x th2) whether all of them are.
struct Done {
    unsigned long long *bits;
    uint8_t *all;
    int tw, th, tw2, th2;
};

// one block per coarse tile, a warp per row of its fine tiles: a pixel is done when its
// closest hit is nearer than every bound from sorted position `at` on (none when skeys is null)
__global__ void __launch_bounds__(256) k_done(const unsigned long long *keys, int W, int H, Done done,
                                              const unsigned long long *skeys, int at) {
    const uint32_t least = skeys ? (uint32_t)(__ldg(&skeys[at]) << 15) : 0u;
    const int lane = threadIdx.x & 31, ty = blockIdx.y * 8 + (threadIdx.x >> 5);
    bool all = true;
#pragma unroll
    for (int k = 0; k < 8; k++) {
        const int tx = blockIdx.x * 8 + k;
        const int i = tx * 8 + (lane & 7), j = ty * 8 + (lane >> 3);
        const bool d0 = i >= W || j >= H || key_dist(__ldcg(&keys[(size_t)j * W + i])) < least;
        const bool d1 = i >= W || j + 4 >= H || key_dist(__ldcg(&keys[(size_t)(j + 4) * W + i])) < least;
        const unsigned m0 = __ballot_sync(0xffffffffu, d0), m1 = __ballot_sync(0xffffffffu, d1);
        if (lane == 0 && tx < done.tw && ty < done.th) done.bits[ty * done.tw + tx] = m0 | ((unsigned long long)m1 << 32);
        all = all && (m0 & m1) == 0xffffffffu;
    }
    const int n = __syncthreads_and(all);
    if (threadIdx.x == 0) done.all[blockIdx.y * done.tw2 + blockIdx.x] = (uint8_t)(n != 0);
}

// true when every pixel of the tiles over the box [i0, i1] x [j0, j1] is done (fine tiles when
// the box spans few of them, else coarse ones)
__device__ bool box_done(const Done &z, int i0, int j0, int i1, int j1) {
    int x0 = i0 >> kTileShift, x1 = i1 >> kTileShift, y0 = j0 >> kTileShift, y1 = j1 >> kTileShift;
    if ((x1 - x0 + 1) * (y1 - y0 + 1) <= kMaxFineTiles) {
        for (int y = y0; y <= y1; y++)
            for (int x = x0; x <= x1; x++)
                if (~__ldg(&z.bits[y * z.tw + x])) return false;
        return true;
    }
    x0 = i0 >> kCoarseShift; x1 = i1 >> kCoarseShift; y0 = j0 >> kCoarseShift; y1 = j1 >> kCoarseShift;
    for (int y = y0; y <= y1; y++)
        for (int x = x0; x <= x1; x++)
            if (!__ldg(&z.all[y * z.tw2 + x])) return false;
    return true;
}

// Setup of every triangle; the small ones are rasterised here, the others queued.
// `split` warps serve each group of 32 triangles (each sets the group up and takes every
// split-th stretch of 32 of its candidate pixels), so that scenes with few triangles
// still occupy the GPU.  They must agree on the list: nothing writes the done bits meanwhile.
__global__ void __launch_bounds__(kRastThreads) k_rast_small(DevCam cam, SceneDev sc, const uint32_t *order,
                                                              int count, int split, const float *tnear, Done done,
                                                              unsigned long long *keys, BigTri *big, int max_big,
                                                              Cut cut, uint32_t *chunk_start, BigCounts *counts) {
    __shared__ SmallSlot slot[kRastThreads];
    __shared__ int excl[kRastThreads];
    const int lane = threadIdx.x & 31, wbase = threadIdx.x & ~31;
    const int gw = blockIdx.x * (kRastThreads / 32) + (threadIdx.x >> 5);
    const int part = gw % split;
    const int idx = (gw / split) * 32 + lane;
    const int k = idx < count ? (int)__ldg(&order[idx]) : 0;
    int npx = 0;
    if (idx < count) {
        const float4 *tp = sc.tris + 3 * (size_t)k;
        const float4 v0 = __ldg(tp), v1 = __ldg(tp + 1), v2 = __ldg(tp + 2);
        TriSetup S;
        const float tn = __ldg(&tnear[k]);
        if (tri_setup(cam, v0, v1, v2, S) && !box_done(done, S.i0, S.j0, S.i1, S.j1)) {
            const int bw = S.i1 - S.i0 + 1, bh = S.j1 - S.j0 + 1;
            const long long n = (long long)bw * bh;
            if (n > kSmallPx) {
                if (part == 0) {                     // the group's first warp queues it
                    BigTri B;
                    B.e0 = make_float4(S.e[0], S.e[1], S.e[2], 0.f);
                    B.e1 = make_float4(S.e[3], S.e[4], S.e[5], 0.f);
                    B.e2 = make_float4(S.e[6], S.e[7], S.e[8], 0.f);
                    B.box = make_int4(S.i0, S.j0, S.i1, S.j1);
                    B.k = k;
                    B.tn = tn;
                    B.tiles = ((S.i1 >> kTileShift) - (S.i0 >> kTileShift) + 1) * ((S.j1 >> kTileShift) - (S.j0 >> kTileShift) + 1);
                    B.pad = 0;
                    // one warp's work from the front of the queue; what is cut into chunks from
                    // its end, its place and its first chunk from one atomic, so that the first
                    // chunks ascend with the places
                    if (B.tiles <= cut.tiles) {
                        big[atomicAdd(&counts->one, 1u)] = B;
                    } else {
                        const uint32_t per = cut.per_chunk(B.tiles), n_chunks = ((uint32_t)B.tiles + per - 1u) / per;
                        const unsigned long long at = atomicAdd(&counts->cut, (1ull << 32) | n_chunks);
                        big[(uint32_t)max_big - 1u - (uint32_t)(at >> 32)] = B;
                        chunk_start[at >> 32] = (uint32_t)at;
                    }
                }
            } else {
                npx = (int)n;
                SmallSlot &o = slot[threadIdx.x];
#pragma unroll
                for (int q = 0; q < 9; q++) o.e[q] = S.e[q];
                o.i0 = S.i0; o.j0 = S.j0; o.bw = bw; o.rbw = 1.f / (float)bw;
                o.tn = tn;
                o.v0 = v0; o.v1 = v1; o.v2 = v2;
            }
        }
    }
    // the warp's candidate pixels as one list
    int incl = npx;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += v;
    }
    const int total = __shfl_sync(0xffffffffu, incl, 31);
    excl[threadIdx.x] = incl - npx;
    __syncwarp();
    for (int w = lane + 32 * part; w < total; w += 32 * split) {
        // owner: the last triangle whose list starts at or before w (it has pixels)
        int l = 0;
#pragma unroll
        for (int step = 16; step; step >>= 1)
            if (excl[wbase + l + step] <= w) l += step;
        const SmallSlot &o = slot[wbase + l];
        int q, r;
        divmod(w - excl[wbase + l], o.bw, o.rbw, q, r);
        const int i = o.i0 + r, j = o.j0 + q;
        if (edges_pass(o.e, i + 0.5f, j + 0.5f) && !occluded(keys, (size_t)j * cam.W + i, o.tn))
            test_pixel(cam, keys, i, j, o.v0, o.v1, o.v2);
    }
}

// A warp's working lists: tiles to cover (the triangle's place in the queue and the tile), the
// pixels that 32 tiles leave (lane of the tile << 6 | pixel of the tile), and the pixels whose
// closest hit so far the triangle may beat.
struct RastWarp {
    uint32_t tri[64];
    int tile[64];
    uint16_t px[32 * 64];
    uint32_t test_tri[64];
    int2 test_ij[64];
};

// the ray tests of the last n (<= 32) listed pixels, one per lane
__device__ __forceinline__ void test_listed(const DevCam &cam, const SceneDev &sc, unsigned long long *keys,
                                            const BigTri *__restrict__ big, const RastWarp &Q, int first, int n, int lane) {
    if (lane < n) {
        const int2 ij = Q.test_ij[first + lane];
        const float4 *tp = sc.tris + 3 * (size_t)__ldg(&big[Q.test_tri[first + lane]].k);
        test_pixel(cam, keys, ij.x, ij.y, __ldg(tp), __ldg(tp + 1), __ldg(tp + 2));
    }
    __syncwarp();
}

// Up to 32 queued tiles, one per lane: the pixels that pass the three edges (edges_pass,
// evaluated for all 64 pixels of the tile), lie in the triangle's box and are not done.  They
// form one list, which the lanes check against the pixels' closest hits 32 at a time; what is
// left is listed again (`tests` entries wait on entry and exit) and gets its ray tests 32 at a
// time, so that the long test runs with all its lanes.
__device__ __forceinline__ void cover_tiles(const DevCam &cam, const SceneDev &sc, unsigned long long *keys, const Done &done,
                                            const BigTri *__restrict__ big, RastWarp &Q, int first, int n, int lane, int &tests) {
    unsigned long long mask = 0ull;
    uint32_t tri = 0;
    int tx = 0, ty = 0;
    float tn = 0.f;
    if (lane < n) {
        tri = Q.tri[first + lane];
        const int tile = Q.tile[first + lane];
        ty = tile / done.tw;
        tx = tile - ty * done.tw;
        const BigTri &B = big[tri];
        const float4 e0 = __ldg(&B.e0), e1 = __ldg(&B.e1), e2 = __ldg(&B.e2);
        const int4 box = __ldg(&B.box);
        tn = __ldg(&B.tn);
        const float x0 = (float)(tx * 8) + 0.5f, y0 = (float)(ty * 8) + 0.5f;
        unsigned half[2];
#pragma unroll
        for (int h = 0; h < 2; h++) {
            unsigned out = 0u;                       // bit = 1: an edge is negative
#pragma unroll
            for (int r = 3; r >= 0; r--) {
                const float y = y0 + (float)(4 * h + r);
                const float c0 = fmaf(e0.y, y, e0.z), c1 = fmaf(e1.y, y, e1.z), c2 = fmaf(e2.y, y, e2.z);
#pragma unroll
                for (int k = 7; k >= 0; k--) {
                    const float x = x0 + (float)k;
                    const float m = fminf(fminf(fmaf(e0.x, x, c0), fmaf(e1.x, x, c1)), fmaf(e2.x, x, c2));
                    out = (out << 1) | (m >= 0.f ? 0u : 1u);
                }
            }
            half[h] = ~out;
        }
        mask = half[0] | ((unsigned long long)half[1] << 32);
        // the box's columns and rows in the tile
        const int cl = max(box.x - tx * 8, 0), cr = min(box.z - tx * 8, 7), rl = max(box.y - ty * 8, 0), rr = min(box.w - ty * 8, 7);
        const unsigned long long col = ((0xffu << cl) & (0xffu >> (7 - cr)) & 0xffu) * 0x0101010101010101ull;
        const unsigned long long row = (~0ull << (8 * rl)) & (~0ull >> (8 * (7 - rr)));
        mask &= col & row & ~__ldg(&done.bits[tile]);
    }
    // the pixels as one list
    const int np = __popcll(mask);
    int incl = np;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += v;
    }
    const int total = __shfl_sync(0xffffffffu, incl, 31);
    int at = incl - np;
#pragma unroll
    for (int h = 0; h < 2; h++)
        for (unsigned m = h ? (unsigned)(mask >> 32) : (unsigned)mask; m; m &= m - 1)
            Q.px[at++] = (uint16_t)((lane << 6) | (32 * h + __ffs(m) - 1));
    __syncwarp();
    const unsigned lt = (1u << lane) - 1u;
    for (int w = 0; w < total; w += 32) {
        const int e = w + lane < total ? Q.px[w + lane] : 0;
        const int o = e >> 6, b = e & 63;
        const uint32_t t = __shfl_sync(0xffffffffu, tri, o);
        const float bound = __shfl_sync(0xffffffffu, tn, o);
        const int i = __shfl_sync(0xffffffffu, tx, o) * 8 + (b & 7), j = __shfl_sync(0xffffffffu, ty, o) * 8 + (b >> 3);
        const bool live = w + lane < total && !occluded(keys, (size_t)j * cam.W + i, bound);
        const unsigned m = __ballot_sync(0xffffffffu, live);
        if (live) {
            const int p = tests + __popc(m & lt);
            Q.test_tri[p] = t;
            Q.test_ij[p] = make_int2(i, j);
        }
        tests += __popc(m);
        __syncwarp();
        if (tests >= 32) {
            tests -= 32;
            test_listed(cam, sc, keys, big, Q, tests, 32, lane);
        }
    }
}

// The queued triangles: warps claim them one at a time, then the chunks of the others.  The
// lanes look at 32 tiles of the box at once and drop a tile when it is finished or when an
// edge is negative at its best corner -- edge_at is monotone in x and in y, roundings
// included, so every pixel of the tile fails the same test.  The others are covered 32 at a
// time, across triangles.
__global__ void __launch_bounds__(kBigThreads) k_rast_big(const __grid_constant__ DevCam cam, const __grid_constant__ SceneDev sc,
                                                           unsigned long long *keys, const __grid_constant__ Done done,
                                                           const BigTri *__restrict__ big, int max_big, Cut cutting,
                                                           const uint32_t *__restrict__ chunk_start, BigCounts *counts) {
    __shared__ RastWarp lists[kBigThreads / 32];
    RastWarp &Q = lists[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    const uint32_t nb = __ldg(&counts->one);
    const unsigned long long cut = __ldg(&counts->cut);
    const uint32_t n_cut = (uint32_t)(cut >> 32);
    const unsigned long long total = (unsigned long long)nb + (uint32_t)cut;
    int queued = 0, tests = 0;
    for (;;) {
        uint32_t c = 0;
        if (lane == 0) c = atomicAdd(&counts->cursor, 1u);
        c = __shfl_sync(0xffffffffu, c, 0);
        if (c >= total) break;
        uint32_t at = c;
        int t0 = 0, t1;
        if (c < nb) {
            t1 = __ldg(&big[at].tiles);
        } else {
            c -= nb;
            // the last triangle whose chunks start at or before c: 32 places looked at per step
            uint32_t lo = 0, n = n_cut;
            while (n > 1) {
                const uint32_t step = (n + 31) / 32, p = lo + (uint32_t)lane * step;
                const bool le = (uint32_t)lane * step < n && __ldg(&chunk_start[p]) <= c;
                const uint32_t k = 31 - __clz(__ballot_sync(0xffffffffu, le));   // lane 0 always is
                n = min(step, n - k * step);
                lo += k * step;
            }
            at = (uint32_t)max_big - 1u - lo;
            const int tiles = __ldg(&big[at].tiles);
            const uint32_t per = cutting.per_chunk(tiles);
            t0 = (int)((c - __ldg(&chunk_start[lo])) * per);
            t1 = min(tiles, t0 + (int)per);
        }
        const BigTri &B = big[at];
        const float4 e0 = __ldg(&B.e0), e1 = __ldg(&B.e1), e2 = __ldg(&B.e2);
        const int4 box = __ldg(&B.box);
        const float e[9] = {e0.x, e0.y, e0.z, e1.x, e1.y, e1.z, e2.x, e2.y, e2.z};
        const int tx0 = box.x >> kTileShift, ty0 = box.y >> kTileShift;
        const int tw = (box.z >> kTileShift) - tx0 + 1;
        const float rtw = 1.f / (float)tw;
        for (int base = t0; base < t1; base += 32) {
            const int t = base + lane;
            int tile = 0;
            bool in = t < t1;
            if (in) {
                int q, r;
                divmod(t, tw, rtw, q, r);
                const int tx = tx0 + r, ty = ty0 + q;
                tile = ty * done.tw + tx;
                // the box's pixel centres in the tile
                const float xl = (float)max(tx * 8, box.x) + 0.5f, xh = (float)min(tx * 8 + 7, box.z) + 0.5f;
                const float yl = (float)max(ty * 8, box.y) + 0.5f, yh = (float)min(ty * 8 + 7, box.w) + 0.5f;
#pragma unroll
                for (int k = 0; k < 3; k++)
                    in = in && edge_at(e + 3 * k, e[3 * k] > 0.f ? xh : xl, e[3 * k + 1] > 0.f ? yh : yl) >= 0.f;
                in = in && ~__ldg(&done.bits[tile]) != 0ull;
            }
            const unsigned m = __ballot_sync(0xffffffffu, in);
            if (in) {
                const int o = queued + __popc(m & lt);
                Q.tri[o] = at;
                Q.tile[o] = tile;
            }
            queued += __popc(m);
            __syncwarp();
            if (queued >= 32) {
                queued -= 32;
                cover_tiles(cam, sc, keys, done, big, Q, queued, 32, lane, tests);
                __syncwarp();
            }
        }
    }
    if (queued > 0) cover_tiles(cam, sc, keys, done, big, Q, 0, queued, lane, tests);
    if (tests > 0) test_listed(cam, sc, keys, big, Q, 0, tests, lane);
}

// closest hit per pixel -> colour, depth, normal, id (as the ray-cast producer writes them)
__global__ void __launch_bounds__(kRastThreads) k_rast_resolve(DevCam cam, DevParams p, SceneDev sc,
                                                                const unsigned long long *keys,
                                                                const int32_t *prim_k, float4 *color, float *depth,
                                                                float4 *normal, int32_t *prim) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y * blockDim.y + threadIdx.y;
    if (i >= cam.W || j >= cam.H) return;
    const size_t q = (size_t)j * cam.W + i;
    const unsigned long long key = keys[q];
    if (key == ~0ull) {
        if (prim) prim[q] = -1;
        color[q] = make_float4(p.sky.x, p.sky.y, p.sky.z, 1.f);
        depth[q] = INFINITY;
        normal[q] = make_float4(0.f, 0.f, 0.f, 0.f);
        return;
    }
    HitRec h;
    h.t = __uint_as_float((uint32_t)(key >> 32));
    h.prim = (int)(uint32_t)key;
    h.k = __ldg(&prim_k[h.prim]);
    const float3 d = pixel_dir(cam, i + 0.5f, j + 0.5f);
    float3 n;
    const float3 col = shade(p, sc, h, d, n);
    if (prim) prim[q] = h.prim;
    color[q] = make_float4(col.x, col.y, col.z, 1.f);
    depth[q] = h.t * dot(d, cam.F);
    normal[q] = make_float4(n.x, n.y, n.z, 0.f);
}

// per triangle: its distance bound, and the sort key (the top 16 of the bound's 31 bits:
// non-negative floats order as unsigned integers, and 1/256 of the distance is order enough)
// with its index
__global__ void k_tri_near(DevCam cam, SceneDev sc, int n_tot, float *tnear, unsigned long long *skeys,
                           uint32_t *svals) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n_tot) return;
    const float4 *tp = sc.tris + 3 * (size_t)k;
    const float tn = near_bound(cam, __ldg(tp), __ldg(tp + 1), __ldg(tp + 2));
    tnear[k] = tn;
    skeys[k] = (unsigned long long)(__float_as_uint(tn) >> 15);
    svals[k] = (uint32_t)k;
}

// inverse of the tree order: triangle id -> sorted index
__global__ void k_prim_index(const float4 *tris, int n, int32_t *prim_k) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < n) prim_k[__float_as_int(__ldg(&tris[3 * (size_t)k]).w)] = k;
}

}  // namespace

void launch_prim_index(const float4 *tris, int n, int32_t *prim_k, cudaStream_t st) {
    if (n > 0) {
        k_prim_index<<<(n + 255) / 256, 256, 0, st>>>(tris, n, prim_k);
        count_launches(1);
    }
}

// ends of the depth-ordered batches: the nearest 1/32, as many again, then twice as many each; scenes under
// kSortedMin triangles run as one batch in scene order (the sort and the launches would cost
// more than they save)
constexpr int kBatches = 6;
constexpr int kSortedMin = 65536;
__host__ inline int batch_end(int b, int nb, int n) { return b + 1 >= nb ? n : (int)((long long)n >> (nb - 1 - b)); }

// Scratch of one call, from the context's stream-ordered pool.
size_t raster_scratch_bytes(int W, int H, int n_tot) {
    auto up = [](size_t b) { return (b + 255) & ~(size_t)255; };
    const size_t n = (size_t)n_tot;
    const size_t t1 = (size_t)((W + 7) >> kTileShift) * ((H + 7) >> kTileShift);
    const size_t t2 = (size_t)((W + 63) >> kCoarseShift) * ((H + 63) >> kCoarseShift);
    return up(8 * (size_t)W * H) + up(sizeof(BigTri) * n) + up(4 * (n + 1)) + up(sizeof(BigCounts) * kBatches) +
           up(4 * n) + 2 * up(8 * n) + 2 * up(4 * n) + up(4 * sort_pairs_scratch_ints(n_tot)) + up(8 * t1) +
           up(t2);
}

cudaError_t launch_raster(const DevCam &cam, const DevParams &p, const SceneDev &sc, const int32_t *prim_k,
                          void *scratch, int sm_count, float4 *color, float *depth, float4 *normal, int32_t *prim,
                          cudaStream_t st) {
    auto up = [](size_t b) { return (b + 255) & ~(size_t)255; };
    const int n_tot = sc.n_tris + sc.n_large;
    char *base = static_cast<char *>(scratch);
    unsigned long long *keys = reinterpret_cast<unsigned long long *>(base);
    base += up(8 * (size_t)cam.W * cam.H);
    BigTri *big = reinterpret_cast<BigTri *>(base);
    base += up(sizeof(BigTri) * (size_t)n_tot);
    uint32_t *chunk_start = reinterpret_cast<uint32_t *>(base);
    base += up(4 * ((size_t)n_tot + 1));
    BigCounts *counts = reinterpret_cast<BigCounts *>(base);
    base += up(sizeof(BigCounts) * kBatches);
    Cut cut;
    cut.tiles = std::min(kChunkTiles, std::max(kChunkTilesFew, n_tot / 1024));
    cut.most = std::min(65536u, std::max(1u, 0x7FFFFFFFu / (uint32_t)std::max(n_tot, 1)));
    const size_t n = (size_t)n_tot;
    float *tnear = reinterpret_cast<float *>(base);
    base += up(4 * n);
    unsigned long long *skeys = reinterpret_cast<unsigned long long *>(base);
    base += up(8 * n);
    unsigned long long *skeys2 = reinterpret_cast<unsigned long long *>(base);
    base += up(8 * n);
    uint32_t *order = reinterpret_cast<uint32_t *>(base);
    base += up(4 * n);
    uint32_t *order2 = reinterpret_cast<uint32_t *>(base);
    base += up(4 * n);
    int *sort_scratch = reinterpret_cast<int *>(base);
    base += up(4 * sort_pairs_scratch_ints(n_tot));
    Done done;
    done.tw = (cam.W + 7) >> kTileShift; done.th = (cam.H + 7) >> kTileShift;
    done.tw2 = (cam.W + 63) >> kCoarseShift; done.th2 = (cam.H + 63) >> kCoarseShift;
    done.bits = reinterpret_cast<unsigned long long *>(base);
    base += up(8 * (size_t)done.tw * done.th);
    done.all = reinterpret_cast<uint8_t *>(base);
    cudaError_t e = cudaMemsetAsync(keys, 0xFF, 8 * (size_t)cam.W * cam.H, st);
    if (e == cudaSuccess) e = cudaMemsetAsync(counts, 0, sizeof(BigCounts) * kBatches, st);
    if (e != cudaSuccess) return e;
    if (n_tot > 0) {
        // the triangles nearest first
        const int nbat = n_tot >= kSortedMin ? kBatches : 1;
        k_tri_near<<<(n_tot + 255) / 256, 256, 0, st>>>(cam, sc, n_tot, tnear, skeys, order);
        if (nbat > 1) sort_pairs_by_low_bits(skeys, order, skeys2, order2, n_tot, 16, sort_scratch, st);
        for (int bt = 0, b0 = 0; bt < nbat; bt++) {
            const int b1 = batch_end(bt, nbat, n_tot);
            if (b1 <= b0) continue;
            BigCounts *cb = counts + bt;
            k_done<<<dim3(done.tw2, done.th2), 256, 0, st>>>(keys, cam.W, cam.H, done, nbat > 1 ? skeys : nullptr, b0);
            // at least 32 warps per SM: groups of 32 triangles are split over several warps
            const int groups = (b1 - b0 + 31) / 32;
            const int split = std::min(16, std::max(1, (32 * sm_count + groups - 1) / groups));
            const int warps = groups * split;
            k_rast_small<<<(warps + kRastThreads / 32 - 1) / (kRastThreads / 32), kRastThreads, 0, st>>>(
                cam, sc, order + b0, b1 - b0, split, tnear, done, keys, big, n_tot, cut, chunk_start, cb);
            k_rast_big<<<8 * sm_count, kBigThreads, 0, st>>>(cam, sc, keys, done, big, n_tot, cut, chunk_start, cb);
            count_launches(3);
            b0 = b1;
        }
        count_launches(1);
    }
    dim3 b(32, 8), g((cam.W + 31) / 32, (cam.H + 7) / 8);
    k_rast_resolve<<<g, b, 0, st>>>(cam, p, sc, keys, prim_k, color, depth, normal, prim);
    count_launches(1);
    return cudaGetLastError();
}
