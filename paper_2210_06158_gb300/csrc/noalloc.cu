// Allocation-free variant of the tile stage of the post-process (tile max-CoC and
// its neighbourhood dilation), for callers that must not allocate device memory.
//
// Some hosts of this library cannot call cudaMalloc at the point where they want the
// tile map: an engine whose allocator has reserved all device memory up front and
// hands out nothing during a frame, or a frame loop in which cudaMalloc/cudaFree
// would implicitly synchronise the device and stall the frame.  This entry point
// keeps its only intermediate -- the per-tile maxima before dilation -- in a
// file-scope __device__ array instead of a buffer it would have to allocate.
//
// The array holds at most kMaxTiles tiles (512 KB).  Every GPU on which the library
// is loaded holds that array for the life of the process.  All calls share it and it
// keeps whatever the previous call left there; each call overwrites every tile it
// reads before reading it, so nothing has to start at zero.  Calls whose work
// overlaps on the GPU (different streams, or different host threads without
// ordering) race on the array and must be serialised by the caller.
#include <math.h>
#include <string.h>

#include "dof_internal.cuh"

namespace {

constexpr int kMaxTiles = DOF_NOALLOC_MAX_TILES;

// the scratch array: raw (undilated) tile maxima (near radius, |rho|)
__device__ __align__(256) float2 g_tile_scratch[kMaxTiles];

struct TileArgs {
    float cocK, d, rmax, z_far;
    int W, H, W2, H2, TW, TH, K;
};

// Tile maxima from the full-resolution depth: depth of a half-resolution pixel = the nearest of
// its 2x2 block (clamped to z_far), rho = clamp(c(z)/4, +-rmax), c(z) = cocK (z - d) / z.
//
// Bound: the read of the depth map (33 MB at 4K, 5 us at the copy rate).  A warp takes a strip of
// four 8x8 tiles, a lane one column of its eight rows, so sixteen 8-byte loads per lane are
// in flight before the first is used; a block per tile of one load each took 18 us at 4K, this
// 5.6 us.
__global__ void __launch_bounds__(128) k_tiles_scratch(const __grid_constant__ TileArgs a, const float *__restrict__ depth,
                                                       float2 *raw) {
    const int lane = threadIdx.x & 31, ty = blockIdx.y;
    const int tx0 = (blockIdx.x * 4 + (int)(threadIdx.x >> 5)) * 4;      // the strip's first tile
    if (tx0 >= a.TW) return;
    const int i = tx0 * 8 + lane;
    float2 d[8][2];
#pragma unroll
    for (int r = 0; r < 8; r++) {
        const int j = ty * 8 + r;
        const bool in = i < a.W2 && j < a.H2;
        const size_t f = in ? (size_t)(2 * j) * a.W + 2 * i : 0;
        d[r][0] = __ldg(reinterpret_cast<const float2 *>(&depth[f]));
        d[r][1] = __ldg(reinterpret_cast<const float2 *>(&depth[in ? f + a.W : 0]));
    }
    float nm = 0.f, am = 0.f;
#pragma unroll
    for (int r = 0; r < 8; r++) {
        if (i < a.W2 && ty * 8 + r < a.H2) {
            const float z = fminf(fminf(fminf(d[r][0].x, a.z_far), fminf(d[r][0].y, a.z_far)),
                                  fminf(fminf(d[r][1].x, a.z_far), fminf(d[r][1].y, a.z_far)));
            const float rho = fminf(fmaxf(0.25f * (a.cocK * (z - a.d) / z), -a.rmax), a.rmax);
            nm = fmaxf(nm, fmaxf(0.f, -rho));
            am = fmaxf(am, fabsf(rho));
        }
    }
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) {
        nm = fmaxf(nm, __shfl_xor_sync(0xffffffffu, nm, o));
        am = fmaxf(am, __shfl_xor_sync(0xffffffffu, am, o));
    }
    const int tx = tx0 + (lane >> 3);
    if ((lane & 7) == 0 && tx < a.TW) raw[ty * a.TW + tx] = make_float2(nm, am);
}

// Neighbourhood max over (2K+1)^2 tiles, from the scratch array into the caller's map: the
// block's tiles and their halo staged in shared memory, then the maxima of rows, then of
// columns (K <= 16).  2 x (2K+1) shared reads per tile instead of (2K+1)^2 global ones: 8.0 ->
// 2.9 us at 4K (K = 4).
constexpr int kDilW = 32, kDilH = 8, kDilMaxK = 16;
__global__ void __launch_bounds__(kDilW * kDilH) k_dilate_scratch(const __grid_constant__ TileArgs a, const float2 *raw,
                                                                  float2 *dil) {
    __shared__ float2 t[kDilH + 2 * kDilMaxK][kDilW + 2 * kDilMaxK];
    __shared__ float2 rows[kDilH + 2 * kDilMaxK][kDilW];
    const int x0 = blockIdx.x * kDilW - a.K, y0 = blockIdx.y * kDilH - a.K;
    const int w = kDilW + 2 * a.K, h = kDilH + 2 * a.K;
    const int tid = threadIdx.y * kDilW + threadIdx.x;
    for (int e = tid; e < w * h; e += kDilW * kDilH) {
        const int y = e / w, x = e - y * w, gx = x0 + x, gy = y0 + y;
        const bool in = gx >= 0 && gy >= 0 && gx < a.TW && gy < a.TH;
        t[y][x] = in ? raw[gy * a.TW + gx] : make_float2(0.f, 0.f);      // the maxima start from 0
    }
    __syncthreads();
    for (int e = tid; e < kDilW * h; e += kDilW * kDilH) {
        const int y = e / kDilW, x = e - y * kDilW;
        float2 m = t[y][x];
        for (int k = 1; k <= 2 * a.K; k++) {
            const float2 v = t[y][x + k];
            m = make_float2(fmaxf(m.x, v.x), fmaxf(m.y, v.y));
        }
        rows[y][x] = m;
    }
    __syncthreads();
    const int tx = blockIdx.x * kDilW + threadIdx.x, ty = blockIdx.y * kDilH + threadIdx.y;
    if (tx >= a.TW || ty >= a.TH) return;
    float2 m = rows[threadIdx.y][threadIdx.x];
    for (int k = 1; k <= 2 * a.K; k++) {
        const float2 v = rows[threadIdx.y + k][threadIdx.x];
        m = make_float2(fmaxf(m.x, v.x), fmaxf(m.y, v.y));
    }
    dil[ty * a.TW + tx] = m;
}

// Device address of g_tile_scratch in the current device's context.  It is looked up
// on every call, not cached: after cudaDeviceReset, or from another context on the same
// device, the library's device code is loaded afresh and the array moves, so an address
// kept from an earlier call could point at memory that is no longer this array.  The
// lookup enqueues no work; the first one in a context loads the library's device code
// there.
int scratch_for_current_device(float2 **out) {
    void *p = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&p, g_tile_scratch);
    if (e != cudaSuccess || !p) return dof_cuda_check(e, "dof_coc_tiles_noalloc: cudaGetSymbolAddress");
    *out = static_cast<float2 *>(p);
    return DOF_OK;
}

}  // namespace

extern "C" int dof_coc_tiles_noalloc(const float *depth, uint32_t width, uint32_t height, const DofCamera *cam,
                                     const DofParams *p, float *tiles_dil, void *stream) {
    if (!depth || !cam || !p || !tiles_dil)
        return dof_set_error(DOF_ERR_INVALID_ARG, "dof_coc_tiles_noalloc: null argument");
    if (width < 2 || height < 2 || (width & 1) || (height & 1) || width > 16384 || height > 16384)
        return dof_set_error(DOF_ERR_INVALID_ARG, "dof_coc_tiles_noalloc: size must be even, 2..16384");
    if (((uintptr_t)depth % 8) || ((uintptr_t)tiles_dil % 8))
        return dof_set_error(DOF_ERR_INVALID_ARG, "dof_coc_tiles_noalloc: depth and tiles must be 8-byte aligned");
    if (p->tile != 8) return dof_set_error(DOF_ERR_INVALID_ARG, "dof_coc_tiles_noalloc: tile must be 8");
    if (!(p->max_coc_px >= 1.f && p->max_coc_px <= 256.f))
        return dof_set_error(DOF_ERR_INVALID_ARG, "dof_coc_tiles_noalloc: max_coc_px must be in [1, 256]");
    if (!(p->z_far_m > 0.f) || !isfinite(p->z_far_m))
        return dof_set_error(DOF_ERR_INVALID_ARG, "dof_coc_tiles_noalloc: z_far must be finite and > 0");
    if (!(cam->f_m > 0.f) || !(cam->f_number > 0.f) || !(cam->sensor_w_m > 0.f) || !(cam->focus_m > cam->f_m) ||
        !isfinite(cam->f_m) || !isfinite(cam->f_number) || !isfinite(cam->focus_m) || !isfinite(cam->sensor_w_m))
        return dof_set_error(DOF_ERR_INVALID_ARG,
                             "dof_coc_tiles_noalloc: need finite f > 0, N > 0, w_s > 0 and focus > f");
    TileArgs a;
    a.W = (int)width; a.H = (int)height; a.W2 = a.W / 2; a.H2 = a.H / 2;
    a.TW = (a.W2 + 7) / 8; a.TH = (a.H2 + 7) / 8;
    if ((long long)a.TW * a.TH > kMaxTiles)
        return dof_set_error(DOF_ERR_INVALID_ARG,
                             "dof_coc_tiles_noalloc: %ux%u needs %d tiles, more than the %d of the built-in scratch",
                             width, height, a.TW * a.TH, kMaxTiles);
    double f = cam->f_m, N = cam->f_number, d = cam->focus_m, ws = cam->sensor_w_m;
    a.cocK = (float)((f / N) * f * (double)width / (ws * (d - f)));
    a.d = cam->focus_m;
    a.rmax = 0.5f * p->max_coc_px;
    a.z_far = p->z_far_m;
    a.K = (int)ceil(0.5 * (double)p->max_coc_px / 8.0);
    float2 *scratch = nullptr;
    int rc = scratch_for_current_device(&scratch);
    if (rc) return rc;
    cudaGetLastError();
    cudaStream_t st = (cudaStream_t)stream;
    k_tiles_scratch<<<dim3((a.TW + 15) / 16, a.TH), 128, 0, st>>>(a, depth, scratch);
    k_dilate_scratch<<<dim3((a.TW + kDilW - 1) / kDilW, (a.TH + kDilH - 1) / kDilH), dim3(kDilW, kDilH), 0, st>>>(
        a, scratch, reinterpret_cast<float2 *>(tiles_dil));
    count_launches(2);
    return dof_cuda_check(cudaGetLastError(), "dof_coc_tiles_noalloc launch");
}
