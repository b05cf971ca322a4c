// lbm_step_noalloc: one time step that allocates no memory, for callers that
// cannot allocate device memory themselves.  One kernel takes the densities, collides
// and pushes (periodic x, half-way bounce-back), on dense FP32 population arrays that the
// caller owns.
//
// The paper has no counterpart: this is an interface for embedding, not part of
// the method.  Same arithmetic as the other FP32 steps (collide.cuh).
#include "collide.cuh"

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <mutex>
#include <string>

namespace lbm {
namespace {

constexpr int kNoAllocMaxSites = 1 << 20;     // largest nx * ny accepted
constexpr int kNoAllocMaxRows = 65535;        // most rows accepted
constexpr int kNoAllocMaxDevices = 64;
constexpr int kCols = 128;                    // columns per block, one per thread

std::mutex g_noalloc_mu;
int g_noalloc_slots[kNoAllocMaxDevices] = {};   // resident blocks of the kernel, by device; 0: not known yet

// The populations (A, B) of site k; n sites per plane.
__device__ __forceinline__ void load_pops(const float* __restrict__ S, size_t n, size_t k, float2 f[9]) {
#pragma unroll
    for (int i = 0; i < 9; ++i) f[i] = make_float2(__ldg(S + (size_t)i * n + k), __ldg(S + (size_t)(9 + i) * n + k));
}

// A block owns kCols columns and the by-th of gridDim.y tiles of (nearly) equal height,
// swept bottom up: the populations of its columns' row y and the densities (B, A) of rows
// y - 1 .. y + 1, with one halo column each side, in a ring in shared memory.  The input
// holds post-streaming populations, so a row's densities are local sums and the next row's
// loads are issued before row y collides.
//
// Bound by latency: one launch and one wave of tiles of a few rows.  The two launches it
// replaces, a density pass and one that collided, read the populations twice.  512x1024,
// whose arrays (75 MB) fit in the L2: 25.1 us before and 16.3 now where they lie in it, 26.4
// and 22.6 where they come from HBM (11.1 us for the 144 bytes per site at the copy rate).
// Loading row y + 2 ahead in a third set of registers measured 15.1 against 16.3, and 36.2
// against 34.7 at 1024x1024.
__global__ void __launch_bounds__(kCols, 5)
noalloc_step_kernel(const float* __restrict__ S, float* __restrict__ out, Physics ph, int nx, int ny) {
    __shared__ float2 sR[4][kCols + 2];
    const int t = threadIdx.x;
    const int x0 = blockIdx.x * kCols;
    const int w = min(kCols, nx - x0);
    const int x = x0 + min(t, w - 1);   // threads past the grid repeat its last column and store nothing
    const bool active = t < w;
    const int y0 = (int)(((long long)blockIdx.y * ny) / gridDim.y);
    const int y1 = (int)(((long long)(blockIdx.y + 1) * ny) / gridDim.y);
    const size_t n = (size_t)nx * ny;
    const int xm = x == 0 ? nx - 1 : x - 1, xp = x == nx - 1 ? 0 : x + 1;
    // threads 64 / 65: the halo columns x0 - 1 / x0 + w
    const bool halo = t == 64 || t == 65;
    const int hx = t == 64 ? (x0 == 0 ? nx - 1 : x0 - 1) : (x0 + w == nx ? 0 : x0 + w);
    const int hs = t == 64 ? 0 : w + 1;

    // densities of row y, populations f, into the ring (zero on the virtual wall rows)
    auto densities = [&](int y, const float2 f[9]) {
        const bool real = y >= 0 && y < ny;
        if (active) sR[y & 3][t + 1] = real ? swap2(sum9_2(f)) : splat(0.0f);
        if (halo) {
            float2 h[9];
            if (real) load_pops(S, n, (size_t)y * nx + hx, h);
            sR[y & 3][hs] = real ? swap2(sum9_2(h)) : splat(0.0f);
        }
    };
    float2 cur[9], nxt[9];
    if (y0 > 0) load_pops(S, n, (size_t)(y0 - 1) * nx + x, nxt);
    load_pops(S, n, (size_t)y0 * nx + x, cur);
    densities(y0 - 1, nxt);
    densities(y0, cur);
#pragma unroll 1
    for (int y = y0; y < y1; ++y) {
        if (y + 1 < ny) load_pops(S, n, (size_t)(y + 1) * nx + x, nxt);
        densities(y + 1, nxt);
        __syncthreads();
        if (active) {
            const float2 *r0 = sR[(y - 1) & 3] + t + 1, *r1 = sR[y & 3] + t + 1, *r2 = sR[(y + 1) & 3] + t + 1;
            Nbr2 p;
            p.E = r1[1]; p.W = r1[-1];
            p.N = r2[0]; p.NE = r2[1]; p.NW = r2[-1];
            p.S = r0[0]; p.SE = r0[1]; p.SW = r0[-1];
            collide_site<true, true>(cur, sum9_2(cur), p, ph, y, ny);
            const size_t k = (size_t)y * nx + x;
#pragma unroll
            for (int i = 0; i < 9; ++i) {
                const int ty = y + cy(i);
                size_t dst = (size_t)opp(i) * n + k;
                if (ty >= 0 && ty < ny) {
                    const int tx = cx(i) == 0 ? x : (cx(i) == 1 ? xp : xm);
                    dst = (size_t)i * n + (size_t)ty * nx + tx;
                }
                out[dst] = cur[i].x;
                out[9 * n + dst] = cur[i].y;
            }
        }
#pragma unroll
        for (int i = 0; i < 9; ++i) cur[i] = nxt[i];
    }
}

lbm_status noalloc_fail(lbm_status st, const std::string& msg) {
    set_last_error(msg);
    return st;
}

}  // namespace
}  // namespace lbm

extern "C" lbm_status lbm_step_noalloc(const lbm_params* p, const float* pops_in, float* pops_out,
                                       void* cuda_stream) {
    using namespace lbm;
    if (!p || !pops_in || !pops_out) return noalloc_fail(LBM_EINVAL, "lbm_step_noalloc: NULL argument");
    if (pops_in == pops_out) return noalloc_fail(LBM_EINVAL, "lbm_step_noalloc: pops_in and pops_out must differ");
    if (p->nx < 4 || p->ny < 8) return noalloc_fail(LBM_EINVAL, "lbm_step_noalloc: nx must be >= 4 and ny >= 8");
    if (p->ny > kNoAllocMaxRows)
        return noalloc_fail(LBM_EINVAL, "lbm_step_noalloc: ny = " + std::to_string(p->ny) + " exceeds " +
                                            std::to_string(kNoAllocMaxRows) + " rows");
    if ((int64_t)p->nx * p->ny > kNoAllocMaxSites)
        return noalloc_fail(LBM_EINVAL, "lbm_step_noalloc: nx * ny = " + std::to_string((int64_t)p->nx * p->ny) +
                                            " exceeds the limit of " + std::to_string(kNoAllocMaxSites) +
                                            " sites; use lbm_step on a handle");
    if (p->storage != LBM_STORE_F32) return noalloc_fail(LBM_EINVAL, "lbm_step_noalloc: FP32 populations only");
    {
        const uintptr_t bytes = (uintptr_t)18 * (uintptr_t)p->nx * (uintptr_t)p->ny * sizeof(float);
        const uintptr_t a = (uintptr_t)pops_in, b = (uintptr_t)pops_out;
        if (a < b + bytes && b < a + bytes)
            return noalloc_fail(LBM_EINVAL, "lbm_step_noalloc: pops_in and pops_out overlap");
    }
    if (!(p->tau_A > 0.5) || !(p->tau_B > 0.5)) return noalloc_fail(LBM_EINVAL, "lbm_step_noalloc: tau must be > 0.5");
    if (p->gravity_mode < 0 || p->gravity_mode > 1)
        return noalloc_fail(LBM_EINVAL, "lbm_step_noalloc: gravity_mode must be 0 or 1");
    if (p->wall_mode < 0 || p->wall_mode > 1)
        return noalloc_fail(LBM_EINVAL, "lbm_step_noalloc: wall_mode must be 0 or 1");
    const double vals[] = {p->G, p->G_wall_A, p->G_wall_B, p->g, p->gx};
    for (double v : vals)
        if (!std::isfinite(v)) return noalloc_fail(LBM_EINVAL, "lbm_step_noalloc: parameters must be finite");

    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return noalloc_fail(LBM_ECUDA, std::string("cudaGetDevice: ") + cudaGetErrorString(e));
    if (dev < 0 || dev >= kNoAllocMaxDevices) return noalloc_fail(LBM_EINVAL, "lbm_step_noalloc: device index too large");
    cudaStream_t st = (cudaStream_t)cuda_stream;
    // an error left by the caller's earlier work is reported, not cleared or taken as ours
    e = cudaPeekAtLastError();
    if (e != cudaSuccess)
        return noalloc_fail(LBM_ECUDA, std::string("lbm_step_noalloc: a CUDA error was pending before the call: ") +
                                           cudaGetErrorString(e));
    cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
    e = cudaStreamIsCapturing(st, &capture);
    if (e != cudaSuccess) return noalloc_fail(LBM_ECUDA, std::string("cudaStreamIsCapturing: ") + cudaGetErrorString(e));
    const int nx = p->nx, ny = p->ny;
    int slots = 0;
    {
        // the device's resident block slots, looked up by the first call outside a capture
        std::lock_guard<std::mutex> lock(g_noalloc_mu);
        slots = g_noalloc_slots[dev];
        if (slots == 0) {
            if (capture != cudaStreamCaptureStatusNone)
                return noalloc_fail(LBM_ESTATE, "lbm_step_noalloc: the first call on a device must come before any stream capture");
            int sms = 0, occ = 0;
            e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
            if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, noalloc_step_kernel, kCols, 0);
            if (e != cudaSuccess) return noalloc_fail(LBM_ECUDA, std::string("lbm_step_noalloc: occupancy: ") + cudaGetErrorString(e));
            slots = g_noalloc_slots[dev] = std::max(1, sms * occ);
        }
    }

    Physics ph;
    ph.tau[0] = (float)p->tau_A;
    ph.tau[1] = (float)p->tau_B;
    ph.om[0] = (float)(1.0 / p->tau_A);
    ph.om[1] = (float)(1.0 / p->tau_B);
    ph.G = (float)p->G;
    ph.ay_wall_bottom[0] = (float)(p->G_wall_A / 6.0);
    ph.ay_wall_bottom[1] = (float)(p->G_wall_B / 6.0);
    ph.ay_wall_top[0] = (float)(-p->G_wall_A / 6.0);
    ph.ay_wall_top[1] = (float)(-p->G_wall_B / 6.0);
    ph.ay_ext[0] = (float)(-p->g);
    ph.ay_ext[1] = (float)(p->gravity_mode == 0 ? p->g : -p->g);
    ph.ax_ext = (float)p->gx;
    ph.wall_mirror = p->wall_mode == 1 ? 1 : 0;
    ph.shift[0] = ph.shift[1] = 0.0f;
    ph.rho_floor[0] = ph.rho_floor[1] = 0.0f;
    ph.step_in = nullptr;
    ph.step_out = nullptr;

    // one wave of tiles, as short as that allows
    const int gx = (nx + kCols - 1) / kCols;
    const int rows = (ny + std::max(1, slots / gx) - 1) / std::max(1, slots / gx);
    noalloc_step_kernel<<<dim3(gx, (ny + rows - 1) / rows), kCols, 0, st>>>(pops_in, pops_out, ph, nx, ny);
    e = cudaGetLastError();
    if (e != cudaSuccess) return noalloc_fail(LBM_ECUDA, std::string("lbm_step_noalloc: step kernel launch: ") + cudaGetErrorString(e));
    return LBM_OK;
}
