// Time-step kernels of the two-component D2Q9 Shan-Chen solver (Section 2 of
// arXiv 2101.04847): pull streaming with periodic x and half-way bounce-back
// walls, densities and common velocity (Eq. 1), Shan-Chen + wall + buoyancy
// accelerations, forced BGK collision with the shifted-velocity equilibrium.
//
// Storage convention.  A buffer B holds *post-collision* populations; the
// post-streaming populations of the kinetic equation are obtained by pulling:
//     S_i(x, y) = B_i(x - c_ix, y - c_iy)   if 0 <= y - c_iy < ny
//     S_i(x, y) = B_opp(i)(x, y)            otherwise (bounce-back at the wall)
// Layout: [direction][y][pitch] cells of both components (lattice.cuh), x fastest.
#include <algorithm>
#include <type_traits>

#include "collide.cuh"

namespace lbm {

__device__ __forceinline__ float2 shift_of(const Physics& ph) { return make_float2(ph.shift[0], ph.shift[1]); }
// FP32 keeps the increments the stored values received (collide_site<true>)
template <typename T> struct Exact { static constexpr bool value = !IsShifted<T>::value; };

// The eight neighbours of ring column c from the density rows S, C, N.
__device__ __forceinline__ Nbr2 ring_nbr(const float2* S, const float2* C, const float2* N, int c) {
    Nbr2 p;
    p.E = C[c + 1]; p.W = C[c - 1];
    p.N = N[c]; p.NE = N[c + 1]; p.NW = N[c - 1];
    p.S = S[c]; p.SE = S[c + 1]; p.SW = S[c - 1];
    return p;
}

// Programmatic dependent launch: a step's blocks may become resident while the step
// before it drains; they wait here, before their first access to global memory, until
// that step has completed and its writes are visible.
__device__ __forceinline__ void wait_previous_step() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// ---------------------------------------------------------------------------
// Fused pull stream-collide.  A block owns kThreadsX columns and tile_y rows and
// sweeps its rows bottom-up.  Each thread keeps the populations of its column for
// the current and the next row in registers; the densities of three consecutive
// rows (plus one halo column each side), as (B, A), live in a 4-slot shared-memory
// ring.  The only redundant loads are the pulls of the halo columns and of the two
// halo rows y0 - 1 and y1, which only feed densities.
// ---------------------------------------------------------------------------
template <typename T>
__global__ void __launch_bounds__(kThreadsX)
step_fused_kernel(const Cell<T>* __restrict__ fin, Cell<T>* __restrict__ fout, Grid g, Physics ph, int tile_y, int* flag) {
    __shared__ float2 sR[4][kThreadsX + 2];
    const int t = threadIdx.x;
    const uint32_t seed = launch_seed(ph);
    advance_step(ph, blockIdx.x == 0 && blockIdx.y == 0 && t == 0);
    const int x0 = blockIdx.x * kThreadsX;
    const int w = min(kThreadsX, g.nx - x0);
    const int y0 = blockIdx.y * tile_y;
    const int y1 = min(y0 + tile_y, g.ny);
    const bool active = t < w;
    const int x = x0 + (active ? t : w - 1);
    const int xm = x == 0 ? g.nx - 1 : x - 1;
    const int xp = x == g.nx - 1 ? 0 : x + 1;
    // halo columns: left one pulled by thread 0, right one by thread max(w-1, 1)
    const bool haloL = (t == 0);
    const bool haloR = (t == max(w - 1, 1));
    const int hx = haloL ? (x0 == 0 ? g.nx - 1 : x0 - 1) : ((x0 + w) % g.nx);
    const int hxm = hx == 0 ? g.nx - 1 : hx - 1;
    const int hxp = hx == g.nx - 1 ? 0 : hx + 1;
    const int hk = haloL ? 0 : w + 1;
    const bool halo = haloL || haloR;
    const float2 shift = shift_of(ph);

    // row yo into f and its densities into the ring (zero on the virtual wall rows)
    auto pull_row = [&](int yo, float2 f[9]) {
        const int slot = yo & 3;
        float2 r = splat(0.0f), h = splat(0.0f);
        if (yo >= 0 && yo < g.ny) {
            pull_site<T>(fin, g, shift, yo, x, xm, xp, f);
            r = swap2(sum9_2(f));
            if (halo) {
                float2 tmp[9];
                pull_site<T>(fin, g, shift, yo, hx, hxm, hxp, tmp);
                h = swap2(sum9_2(tmp));
            }
        }
        if (active) sR[slot][t + 1] = r;
        if (halo) sR[slot][hk] = h;
    };
    float2 cur[9], nxt[9];
    pull_row(y0 - 1, nxt);
    pull_row(y0, cur);
    for (int y = y0; y < y1; ++y) {
        pull_row(y + 1, nxt);
        __syncthreads();
        if (active) {
            const Nbr2 p = ring_nbr(sR[(y - 1) & 3], sR[y & 3], sR[(y + 1) & 3], t + 1);
            if (!collide_site<Exact<T>::value, true>(cur, sum9_2(cur), p, ph, y, g.ny)) atomicOr(flag, 1);
            store_step<T>(fout, g, y, x, cur, shift, seed);
        }
#pragma unroll
        for (int i = 0; i < 9; ++i) cur[i] = nxt[i];
    }
}

// ---------------------------------------------------------------------------
// Staged fused pull stream-collide, one independent sweep per warp.
//
// A warp owns 30 columns [xw, xw + 30) and tile_y rows; lane l handles column
// xw - 1 + l, so lanes 0 and 31 only supply the halo densities of their
// neighbours.  The warp brings its input rows into its own shared-memory ring
// with bulk asynchronous copies (cp.async.bulk, one mbarrier per stage, issued by
// lane 0): row r of all 9 planes, a 16-byte aligned window of kWinW(T) columns
// covering [xw - 2, xw + 32), lands in stage (q0 + r - rfirst) mod kStages.  The
// densities of rows y-1, y, y+1 stay in registers and the x-neighbours come by
// warp shuffles, so no block-wide barrier is ever needed; a warp refills a stage
// after __syncwarp() once all its lanes have read it.  Three input rows are in
// flight ahead of the three in use.
// ---------------------------------------------------------------------------
constexpr int kStages = 6;     // rows y..y+2 in use + 3 rows prefetched
constexpr int kWarpOwned = 30;
constexpr int kWarpsPerBlock = kThreadsX / 32;
constexpr uint32_t kWaitLimit = 1u << 22;
constexpr uint32_t kTestWaitLimit = 4096;   // the timeout test's
template <typename T> struct WinW { static constexpr int value = 40; };   // 36 columns and the alignment slack, 16-byte multiple

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_fence_init() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(smem_addr(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
// Bounded wait: gives up after `limit` polls (kWaitLimit by default) and raises bit 2
// of the guard flag.
__device__ __forceinline__ void mbar_wait(uint64_t* bar, uint32_t parity, int* flag, uint32_t limit = kWaitLimit) {
    for (uint32_t it = 0; it < limit; ++it)
        if (mbar_try_wait(bar, parity)) return;
    atomicOr(flag, 2);
}
__device__ __forceinline__ void bulk_copy_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     smem_addr(dst)),
                 "l"(src), "r"(bytes), "r"(smem_addr(bar))
                 : "memory");
}
__device__ __forceinline__ void fence_proxy_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// Dynamic shared memory of one warp: kStages mbarriers, then the row ring.
template <typename T>
__host__ __device__ constexpr size_t warp_smem_bytes() {
    return 128 + (size_t)kStages * 9 * WinW<T>::value * sizeof(Cell<T>);
}
template <typename T>
size_t warp_kernel_smem_bytes() { return kWarpsPerBlock * warp_smem_bytes<T>(); }

// Post-streaming cells of window column k on row yo from the stages holding rows
// yo-1 (S), yo (C) and yo+1 (N), W columns per plane; on the wall rows the
// populations coming from outside are the bounced-back ones of row yo.
template <int W, typename C>
__device__ __forceinline__ void pull_cells(const C* __restrict__ stS, const C* __restrict__ stC, const C* __restrict__ stN,
                                           bool bottom, bool top, int k, C f[9]) {
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        if (cy(i) == 0) f[i] = stC[i * W + k - cx(i)];
        else if (cy(i) == 1) f[i] = bottom ? stC[opp(i) * W + k] : stS[i * W + k - cx(i)];
        else f[i] = top ? stC[opp(i) * W + k] : stN[i * W + k - cx(i)];
    }
}
// the same as populations
template <typename T, int W>
__device__ __forceinline__ void pull_staged(const Cell<T>* __restrict__ stS, const Cell<T>* __restrict__ stC,
                                            const Cell<T>* __restrict__ stN, bool bottom, bool top, int k, float2 shift,
                                            float2 f[9]) {
    Cell<T> c[9];
    pull_cells<W>(stS, stC, stN, bottom, top, k, c);
#pragma unroll
    for (int i = 0; i < 9; ++i) f[i] = cell_pops<T>(c[i], i, shift);
}

// The neighbours of a lane's column from the lanes beside it: own densities, as
// (B, A), of rows y - 1 (rm), y (rc) and y + 1 (rp).
__device__ __forceinline__ float2 shfl_up2(float2 v) {
    return make_float2(__shfl_up_sync(0xffffffffu, v.x, 1), __shfl_up_sync(0xffffffffu, v.y, 1));
}
__device__ __forceinline__ float2 shfl_down2(float2 v) {
    return make_float2(__shfl_down_sync(0xffffffffu, v.x, 1), __shfl_down_sync(0xffffffffu, v.y, 1));
}
__device__ __forceinline__ Nbr2 lane_nbr(float2 rm, float2 rc, float2 rp) {
    Nbr2 p;
    p.S = rm; p.N = rp;
    p.W = shfl_up2(rc); p.E = shfl_down2(rc);
    p.SW = shfl_up2(rm); p.SE = shfl_down2(rm);
    p.NW = shfl_up2(rp); p.NE = shfl_down2(rp);
    return p;
}

// One warp tile (tx, ty): `my` is the warp's shared-memory region.
template <typename T>
__device__ __forceinline__ void warp_tile(const Cell<T>* __restrict__ fin, Cell<T>* __restrict__ fout, const Grid& g,
                                          const Physics& ph, int tile_y, int tx, int ty, unsigned char* my,
                                          uint32_t seed, int* flag) {
    typedef Cell<T> C;
    constexpr int W = WinW<T>::value;
    const int lane = threadIdx.x & 31;
    uint64_t* bar = reinterpret_cast<uint64_t*>(my);
    C* stage = reinterpret_cast<C*>(my + 128);
    const int xw = tx * kWarpOwned;
    const int y0 = ty * tile_y;
    const int y1 = min(y0 + tile_y, g.ny);
    const int rfirst = max(y0 - 2, 0);
    const int rlast = min(y1 + 1, g.ny - 1);
    const int x = xw - 1 + lane;
    const bool owner = lane >= 1 && lane <= kWarpOwned && x < g.nx;
    constexpr int kAlign = 16 / (int)sizeof(C);
    const int e0 = g.origin + xw - 2;
    const int slack = e0 % kAlign;
    const int k = lane + 1 + slack;                 // window column of this lane's site
    const C* win = fin + (e0 - slack);
    const float2 shift = shift_of(ph);
    const uint32_t row_bytes = W * sizeof(C);

    if (lane == 0) {
        for (int j = 0; j < kStages; ++j) mbar_init(&bar[j], 1);
        mbar_fence_init();
    }
    __syncwarp();
    int next = rfirst;  // next row to issue (lane 0)
    auto issue = [&](int r) {
        const int j = (r - rfirst) % kStages;
        uint64_t* b = &bar[j];
        mbar_expect_tx(b, 9 * row_bytes);
        C* dst = stage + (size_t)j * 9 * W;
        const C* src = win + (size_t)r * g.pitch;
#pragma unroll 1
        for (int p = 0; p < 9; ++p) bulk_copy_g2s(dst + p * W, src + (size_t)p * g.plane, row_bytes, b);
    };
    if (lane == 0)
        for (; next <= rlast && next < rfirst + kStages; ++next) issue(next);
    auto wait_row = [&](int r) {
        if (r >= rfirst && r <= rlast)
            mbar_wait(&bar[(r - rfirst) % kStages], (uint32_t)(((r - rfirst) / kStages) & 1), flag);
    };
    auto stage_of = [&](int r) -> const C* {
        const int rr = min(max(r, rfirst), rlast);
        return stage + (size_t)((rr - rfirst) % kStages) * 9 * W;
    };
    auto pull_row = [&](int yo, float2 f[9]) {
        pull_staged<T, W>(stage_of(yo - 1), stage_of(yo), stage_of(yo + 1), yo == 0, yo == g.ny - 1, k, shift, f);
    };
    // After the reads of row yo (which used input rows up to yo + 1), input rows
    // <= yo - 1 are no longer needed: refill their stages.
    auto refill = [&](int yo) {
        __syncwarp();
        if (lane == 0) {
            fence_proxy_async_smem();
            for (; next <= rlast && next - kStages <= yo - 1; ++next) issue(next);
        }
    };

    float2 fa[9], fb[9];
    float2 rm = splat(0.0f);   // densities of row y - 1, as (B, A) (zero on the virtual wall row)
    if (y0 > 0) {
        wait_row(y0 - 2); wait_row(y0 - 1); wait_row(y0);
        pull_row(y0 - 1, fb);
        rm = swap2(sum9_2(fb));
    }
    wait_row(y0 - 1); wait_row(y0); wait_row(y0 + 1);
    pull_row(y0, fa);
    float2 rc = swap2(sum9_2(fa));      // row y
    refill(y0);

    auto row = [&](int y, float2 cur[9], float2 nxt[9]) {
        float2 rp = splat(0.0f);        // row y + 1
        if (y + 1 < g.ny) {
            wait_row(y + 2);
            pull_row(y + 1, nxt);
            rp = swap2(sum9_2(nxt));
        }
        refill(y + 1);
        const Nbr2 p = lane_nbr(rm, rc, rp);
        if (owner) {
            if (!collide_site<Exact<T>::value, true>(cur, sum9_2(cur), p, ph, y, g.ny)) atomicOr(flag, 1);
            store_step<T>(fout, g, y, x, cur, shift, seed);
        }
        rm = rc;
        rc = rp;
    };
    for (int y = y0; y < y1; y += 2) {
        row(y, fa, fb);
        if (y + 1 < y1) row(y + 1, fb, fa);
    }
}

template <typename T>
__global__ void __launch_bounds__(kThreadsX, 4)
step_warp_kernel(const Cell<T>* __restrict__ fin, Cell<T>* __restrict__ fout, Grid g, Physics ph, int tile_y,
                   int tiles_x, int tiles, int* flag) {
    extern __shared__ __align__(128) unsigned char dsm[];
    const int warp = threadIdx.x >> 5;
    const int tile = blockIdx.x * kWarpsPerBlock + warp;
    const uint32_t seed = launch_seed(ph);
    advance_step(ph, blockIdx.x == 0 && threadIdx.x == 0);
    if (tile >= tiles) return;                      // whole warp leaves together
    warp_tile<T>(fin, fout, g, ph, tile_y, tile % tiles_x, tile / tiles_x,
                 dsm + (size_t)warp * warp_smem_bytes<T>(), seed, flag);
}

// warp tiles of one grid for the per-warp kernel
int warp_tiles(const Grid& g, int tile_y, int* tiles_x) {
    const int tx = (g.nx + kWarpOwned - 1) / kWarpOwned;
    if (tiles_x) *tiles_x = tx;
    return tx * ((g.ny + tile_y - 1) / tile_y);
}

int default_tile_y() { return 32; }

// ---------------------------------------------------------------------------
// Pipelined fused pull stream-collide.  A block of 4 warps shares one ring of
// input rows (bulk asynchronous copies of all 9 planes, 16-byte aligned windows of
// kPipeWin columns covering [x0 - 2, x0 + 122)); each warp sweeps its own 32 columns
// (30 owned, lanes 0 and 31 supply halo densities) with the x-neighbour densities
// from warp shuffles, so warps never wait for one another at a block barrier.  A
// stage is refilled once all four warps have released its row (an "empty"
// mbarrier per stage, one arrival per warp); warp 0's lane 0 issues the copies,
// blocking only for a row it is about to read itself.
// ---------------------------------------------------------------------------
constexpr int kPipeStages = 5;
constexpr int kPipeOwned = kWarpsPerBlock * kWarpOwned;   // 120 columns per block
constexpr int kPipeWin = 136;                              // >= 124 + 7, 16-byte multiple for 2- and 4-byte types

template <typename T>
__host__ __device__ constexpr size_t pipe_smem_bytes() {
    return 128 + (size_t)kPipeStages * 9 * kPipeWin * sizeof(Cell<T>);
}

__device__ __forceinline__ bool mbar_test(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(smem_addr(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(bar)) : "memory");
}

template <typename T>
__global__ void __launch_bounds__(kThreadsX, 4)
step_pipe_kernel(const Cell<T>* __restrict__ fin, Cell<T>* __restrict__ fout, Grid g, Physics ph, int tile_y, int* flag) {
    typedef Cell<T> C;
    const uint32_t seed = launch_seed(ph);
    advance_step(ph, blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0);
    constexpr int S = kPipeStages;
    extern __shared__ __align__(128) unsigned char dsm[];
    uint64_t* full = reinterpret_cast<uint64_t*>(dsm);
    uint64_t* empty = full + S;
    C* stage = reinterpret_cast<C*>(dsm + 128);
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    const int x0 = blockIdx.x * kPipeOwned;
    const int y0 = blockIdx.y * tile_y;
    const int y1 = min(y0 + tile_y, g.ny);
    const int rfirst = max(y0 - 2, 0);
    const int rlast = min(y1 + 1, g.ny - 1);
    const int x = x0 + warp * kWarpOwned - 1 + lane;
    const bool owner = lane >= 1 && lane <= kWarpOwned && x < g.nx;
    constexpr int kAlign = 16 / (int)sizeof(C);
    const int e0 = g.origin + x0 - 2;
    const int slack = e0 % kAlign;
    const int k = warp * kWarpOwned + lane + 1 + slack;
    const C* win = fin + (e0 - slack);
    const float2 shift = shift_of(ph);
    const uint32_t row_bytes = kPipeWin * sizeof(C);
    const bool producer = threadIdx.x == 0;

    if (producer) {
        for (int j = 0; j < S; ++j) {
            mbar_init(&full[j], 1);
            mbar_init(&empty[j], kWarpsPerBlock);
        }
        mbar_fence_init();
    }
    __syncthreads();   // barriers initialised (the only block barrier)

    int next = rfirst;   // next row to issue (producer)
    // Issue rows up to `want`; a row <= `must` is issued even if that means waiting
    // for its stage to be released.
    auto produce = [&](int must, int want) {
        while (next <= rlast && next <= want) {
            const int j = (next - rfirst) % S;
            const int u = (next - rfirst) / S;
            if (u > 0) {
                const uint32_t par = (uint32_t)((u - 1) & 1);
                if (!mbar_test(&empty[j], par)) {
                    if (next > must) break;
                    mbar_wait(&empty[j], par, flag);
                }
            }
            fence_proxy_async_smem();
            mbar_expect_tx(&full[j], 9 * row_bytes);
            C* dst = stage + (size_t)j * 9 * kPipeWin;
            const C* src = win + (size_t)next * g.pitch;
#pragma unroll 1
            for (int p = 0; p < 9; ++p) bulk_copy_g2s(dst + p * kPipeWin, src + (size_t)p * g.plane, row_bytes, &full[j]);
            ++next;
        }
    };
    auto wait_row = [&](int r) {
        if (r < rfirst || r > rlast) return;
        if (warp == 0) {
            if (producer) produce(r, r + S - 3);
            __syncwarp();
        }
        mbar_wait(&full[(r - rfirst) % S], (uint32_t)(((r - rfirst) / S) & 1), flag);
    };
    auto stage_of = [&](int r) -> const C* {
        const int rr = min(max(r, rfirst), rlast);
        return stage + (size_t)((rr - rfirst) % S) * 9 * kPipeWin;
    };
    auto pull_row = [&](int yo, float2 f[9]) {
        if (yo > 0 && yo < g.ny - 1)
            pull_staged<T, kPipeWin>(stage_of(yo - 1), stage_of(yo), stage_of(yo + 1), false, false, k, shift, f);
        else
            pull_staged<T, kPipeWin>(stage_of(yo - 1), stage_of(yo), stage_of(yo + 1), yo == 0, yo == g.ny - 1, k, shift, f);
    };
    int released = rfirst;   // rows < released have been handed back by this warp
    auto release_upto = [&](int r) {   // this warp no longer reads rows <= r
        __syncwarp();
        for (; released <= r && released <= rlast; ++released)
            if (lane == 0) mbar_arrive(&empty[(released - rfirst) % S]);
    };

    float2 fa[9], fb[9];
    float2 rm = splat(0.0f);
    if (y0 > 0) {
        wait_row(y0 - 2); wait_row(y0 - 1); wait_row(y0);
        pull_row(y0 - 1, fb);
        rm = swap2(sum9_2(fb));
    }
    wait_row(y0 - 1); wait_row(y0); wait_row(y0 + 1);
    pull_row(y0, fa);
    float2 rc = swap2(sum9_2(fa));
    release_upto(y0 - 2);

    auto row = [&](int y, float2 cur[9], float2 nxt[9]) {
        float2 rp = splat(0.0f);
        if (y + 1 < g.ny) {
            wait_row(y + 2);
            pull_row(y + 1, nxt);
            rp = swap2(sum9_2(nxt));
        }
        release_upto(y - 1);
        const Nbr2 p = lane_nbr(rm, rc, rp);
        if (owner) {
            if (!collide_site<Exact<T>::value, true>(cur, sum9_2(cur), p, ph, y, g.ny)) atomicOr(flag, 1);
            store_step<T>(fout, g, y, x, cur, shift, seed);
        }
        rm = rc;
        rc = rp;
    };
    for (int y = y0; y < y1; y += 2) {
        row(y, fa, fb);
        if (y + 1 < y1) row(y + 1, fb, fa);
    }
}

// ---------------------------------------------------------------------------
// Block-staged fused pull stream-collide.  A block of TW threads owns TW columns
// [x0, x0 + TW) and the rows [y0, y1) of one of gridDim.y tiles (the ny rows are
// split evenly over the tiles); thread t handles column x0 + t, and threads 64 and
// 65 also supply the densities of the halo columns x0 - 1 and x0 + TW.  Input rows
// are brought into shared memory by bulk asynchronous copies (cp.async.bulk, one
// mbarrier per stage), one plane per lane of lanes 0-8 of warp 0: a 16-byte aligned
// window of BlockWin<T> columns covering [x0 - 2, x0 + TW + 2) of each of the 9 planes a
// row's pull reads (TileRows).  All pulls read shared memory; each input value crosses
// HBM once per tile.  The densities of three rows are exchanged through a shared-memory ring
// (one block barrier per row).
//
// What bounds it: FP32 is limited by HBM (0.97 of the copy rate at 10000x5000, 0.87 at
// 1024x2048, where the ramp of each 51 us launch shows); 16-bit storage by its instructions
// (360 per site with the paired tile below, 57 % of the issue slots: the pipes they share,
// their latency and the row barriers with 16 warps per SM).  Cells of both components halve the loads,
// stores and address arithmetic (FP32 492 -> 361 instructions per site although its tiles
// went from 20 rows to 14, paired FP16 500 -> 360 at 16), a window of TW + 4 FP32 cells needs no alignment slack (34 sectors read per 32
// owned at 128 columns, 36 before), and a tile whose sweep meets no wall row runs code without the wall
// checks.  us per step before and after: FP32 54.0 -> 51.4 (1024x2048), 1232 -> 1094
// (10000x5000); FP16 47.3 -> 36.2, 1024 -> 684; BF16 36.9 -> 27.1 (1501x999).
// ---------------------------------------------------------------------------
// Row stages of a tile (rows y and y + 1 in use, the others prefetched) and the resident
// blocks per SM that its registers are limited for.  FP32 (HBM-bound) is fastest with
// about 800 to 1000 prefetched columns per SM; measured, us per step at 1024x2048 /
// 10000x5000: 128 columns with 3 stages and 6 blocks 51.4 / 1119, 4 and 5 57.0 / 1273,
// 5 and 4 57.0 / 1343; 256 columns with 4 stages and 2 blocks 53.3 / 1101, 3 and 3 52.5 /
// 1145, 5 and 2 57.5 / 1242.
template <typename T, int TW> struct TileCfg {
    static constexpr int kStages = TW == 128 ? 3 : 4, kBlocks = TW == 128 ? 6 : 2;
};
template <int TW> struct TileCfg<__half, TW> { static constexpr int kStages = 5, kBlocks = 768 / TW; };
template <int TW> struct TileCfg<__nv_bfloat16, TW> { static constexpr int kStages = 5, kBlocks = 768 / TW; };

template <typename T, int TW = kBlockTileW> struct BlockWin {
    // TW + 4 columns from x0 - 2 plus the alignment slack of the window start, in
    // 16-byte units; column 0 of a row sits 128 bytes into it and x0 is a multiple of TW
    static constexpr int kAlign = 16 / (int)sizeof(Cell<T>);
    static constexpr int kSlack = (128 / (int)sizeof(Cell<T>) - 2) % kAlign;
    static constexpr int value = (TW + 4 + kSlack + kAlign - 1) / kAlign * kAlign;
};

template <typename T, int TW = kBlockTileW>
__host__ __device__ constexpr size_t block_smem_bytes() {
    return (size_t)TileCfg<T, TW>::kStages * (9 * BlockWin<T, TW>::value * sizeof(Cell<T>) + sizeof(uint64_t));
}

// Density ring of a block tile of TW columns, as (B, A): slot 1 + t holds column
// x0 + t, slots 0 and TW + 1 the halo columns x0 - 1 and x0 + TW.
template <int TW> using BlockRingT = float2[4][TW + 2];

// Planes of row r that the tile [y0, y1) reads (bit i: direction i): all 9 for its
// own rows and the wall rows (bounce-back reads the opposite planes); of the halo
// rows only the populations that stream into the tile or into the density rows y0 - 1
// and y1: c_y = +1 from y0 - 2, c_y = 0 or +1 from y0 - 1, c_y = 0 or -1 from y1 and
// c_y = -1 from y1 + 1 (directions 2, 5, 6 move up, 4, 7, 8 down).
__device__ __forceinline__ uint32_t tile_row_planes(int r, int y0, int y1, int ny) {
    constexpr uint32_t up = (1u << 2) | (1u << 5) | (1u << 6);
    constexpr uint32_t mid = (1u << 0) | (1u << 1) | (1u << 3);
    constexpr uint32_t down = (1u << 4) | (1u << 7) | (1u << 8);
    if ((r >= y0 && r < y1) || r == 0 || r == ny - 1) return up | mid | down;
    if (r == y0 - 2) return up;
    if (r == y0 - 1) return up | mid;
    if (r == y1) return mid | down;
    return down;   // y1 + 1
}

// The densities (A, B) of a site from the sum of its stored values (16-bit storage
// holds h = f - w rho0, whose sum is rho - rho0).
template <typename T>
__device__ __forceinline__ float2 density_of(float2 sum, float2 shift) {
    if constexpr (IsShifted<T>::value) return add2(shift, sum);
    else return sum;
}
template <typename C>
__device__ __forceinline__ float2 sum_cells(const C c[9]) {
    float2 v[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) v[i] = to_f2(c[i]);
    return sum9_2(v);
}
// Collide a site's stored cells (sum: their sum) into the cells to store.
template <typename T, bool kWalls>
__device__ __forceinline__ bool collide_cells(const Cell<T> cur[9], float2 sum, const Nbr2& p, int ny, const Physics& ph,
                                              int y, uint32_t site, uint32_t seed, Cell<T> out[9]) {
    float2 v[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) v[i] = to_f2(cur[i]);
    bool ok;
    if constexpr (IsShifted<T>::value) {
        ok = collide_shifted<kWalls>(v, sum, p, ph, y, ny);
        round_site<T>(site, v, seed, out);
    } else {
        ok = collide_site<true, kWalls>(v, sum, p, ph, y, ny);
#pragma unroll
        for (int i = 0; i < 9; ++i) out[i] = v[i];
    }
    return ok;
}

// The row stages of one tile.  A stage holds what the pull of one row reads: of each
// direction the plane row that streams into it (row r - c_y of direction i for the pull of
// row r, or the row's own opposite plane where that lies beyond a wall), so that a row
// occupies one stage, not the three its source rows would, and every stage is one full
// set of 9 copies.  The pulls are of rows y0 - 1 .. y1, row r in stage (r - y0 + 1) mod S.
// dsm: S stages of 9 planes, then the S mbarriers.
template <typename T, int TW, int S, bool kWithhold>
struct TileRows {
    typedef Cell<T> C;
    static constexpr int W = BlockWin<T, TW>::value;
    static constexpr int kCells = 9 * W;   // per stage
    static constexpr int kStages = S;
    C* stage;
    uint64_t* bar;
    const C* win;   // the window's start in row 0 of plane 0
    size_t plane;
    int y0, y1, ny, pitch;
    int* flag;

    __device__ __forceinline__ TileRows(const C* fin, const Grid& g, int x0, int y0_, int y1_, unsigned char* dsm, int* flag_)
        : plane(g.plane), y0(y0_), y1(y1_), ny(g.ny), pitch(g.pitch), flag(flag_) {
        stage = reinterpret_cast<C*>(dsm);
        bar = reinterpret_cast<uint64_t*>(dsm + (size_t)S * kCells * sizeof(C));
        win = fin + (g.origin + x0 - 2 - BlockWin<T, TW>::kSlack);
        if (threadIdx.x == 0) {
#pragma unroll 1
            for (int j = 0; j < S; ++j) mbar_init(&bar[j], 1);
            mbar_fence_init();
        }
        __syncthreads();
        if (threadIdx.x < 32) {
#pragma unroll 1
            for (int j = 0; j < S; ++j) issue(y0 - 1 + j, j);
        }
    }
    // the pull of row r into stage j (warp 0, all lanes; one direction per lane); a virtual
    // wall row has nothing to copy, its stage's phase completes at once
    __device__ __forceinline__ void issue(int r, int j) {
        if constexpr (kWithhold) return;
        if (r > y1) return;
        const bool real = r >= 0 && r < ny;
        constexpr uint32_t bytes = W * sizeof(C);
        if (threadIdx.x == 0) mbar_expect_tx(&bar[j], real ? 9 * bytes : 0u);
        __syncwarp();
        const int i = threadIdx.x;
        if (i < 9 && real) {
            // directions 2, 5, 6 move up, 4, 7, 8 down
            const int c = (0x64 >> i & 1) - (0x190 >> i & 1);
            const bool inside = r - c >= 0 && r - c < ny;
            const int row = inside ? r - c : r, pl = inside ? i : opp(i);
            bulk_copy_g2s(stage + j * kCells + i * W, win + (size_t)pl * plane + (size_t)row * pitch, bytes, &bar[j]);
        }
    }
    __device__ __forceinline__ void wait_stage(int j, uint32_t phase) {
        mbar_wait(&bar[j], phase, flag, kWithhold ? kTestWaitLimit : kWaitLimit);
    }
};
// Post-streaming cells of window column k from the stage of a row's pull (W columns per
// plane); bounced-back populations come from the column itself.
template <int W, typename C>
__device__ __forceinline__ void pull_stage(const C* __restrict__ st, bool bottom, bool top, int k, C f[9]) {
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        const bool bounced = (cy(i) == 1 && bottom) || (cy(i) == -1 && top);
        f[i] = st[i * W + (bounced ? k : k - cx(i))];
    }
}

// A sweep over the rows of a tile, bottom up, one block barrier per row.
// densities(yo, st): the densities of row yo into the ring, from its stage (yo may be a
// virtual wall row); collide(y, st): row y.  Row y + 1's densities are taken before the
// barrier and row y collided after it, so a row's populations are pulled twice: holding
// them in registers from one iteration to the next instead takes a loop unrolled over
// two rows, whose code (41 KB for the paired tile) outgrew the instruction cache, and 36
// registers.  The two iterations before the tile's first row run without a collision: the
// code stays one copy.
template <typename Rows, typename Densities, typename Collide>
__device__ __forceinline__ void sweep_tile(Rows& R, Densities densities, Collide collide) {
    constexpr int S = Rows::kStages;
    const int y1 = R.y1;
    // pc, pn: the stages of rows y and y + 1; jn that of row y + 1, and the phase of the wait
    // for it, which flips whenever the stage wraps to 0
    const auto *pc = R.stage, *pn = R.stage;
    int jn = 0;
    uint32_t phase = 0;
#pragma unroll 1
    for (int y = R.y0 - 2; y < y1; ++y) {
        R.wait_stage(jn, phase);
        densities(y + 1, pn);
        __syncthreads();
        // every thread is past its reads of rows < y: refill the stage of row y - 1
        if (threadIdx.x < 32 && y >= R.y0) {
            fence_proxy_async_smem();
            R.issue(y - 1 + S, jn >= 2 ? jn - 2 : jn - 2 + S);
        }
        if (y >= R.y0) collide(y, pc);
        pc = pn;
        pn += Rows::kCells;
        if (++jn == S) {
            jn = 0;
            pn = R.stage;
            phase ^= 1u;
        }
    }
}
// Whether a tile's sweep reaches a wall row: its pulls are of rows y0 - 1 .. y1.
__device__ __forceinline__ bool tile_has_walls(int y0, int y1, int ny) { return y0 < 2 || y1 > ny - 2; }

// One block tile: columns [x0, x0 + TW) and rows [y0, y1) of one grid, TW threads.
// dsm: the block_smem_bytes<T, TW>() of dynamic shared memory (row stages, then
// the mbarriers).  kWithhold (the timeout test's instantiation only): no row copy is
// issued and each wait gives up after kTestWaitLimit polls, so every wait of the tile
// runs out with nothing in flight.
template <typename T, int TW, bool kWalls, bool kWithhold>
__device__ __forceinline__ void block_sweep(const Cell<T>* __restrict__ fin, Cell<T>* __restrict__ fout, const Grid& g,
                                            const Physics& ph, int x0, int y0, int y1, unsigned char* dsm,
                                            BlockRingT<TW>& sR, uint32_t seed, int* flag) {
    typedef Cell<T> C;
    constexpr int W = BlockWin<T, TW>::value, slack = BlockWin<T, TW>::kSlack, S = TileCfg<T, TW>::kStages;
    TileRows<T, TW, S, kWithhold> R(fin, g, x0, y0, y1, dsm, flag);
    const int t = threadIdx.x;
    const int x = x0 + t;
    const bool owner = x < g.nx;
    const bool edge = x < 2 || x >= g.nx - 2;
    const int k = t + 2 + slack;
    // threads 64 / 65: the halo columns x0 - 1 / x0 + TW (window columns 1 / TW + 2 + slack)
    const bool halo = t == 64 || t == 65;
    const int kh = t == 64 ? 1 + slack : TW + 2 + slack;
    const int sh = t == 64 ? 0 : TW + 1;
    const float2 shift = shift_of(ph);
    C* q = fout + (size_t)y0 * g.pitch + g.origin + x;
    uint32_t site = site_index(g, y0, x);
    const uint32_t site_row = site_index(g, 1, x) - site_index(g, 0, x);
    bool good = true;
    float2 sum = splat(0.0f), next = splat(0.0f);   // sums of the stored values of rows y, y + 1
    // densities of columns past nx are never read by an owner
    auto densities = [&](int yo, const C* st) {
        float2* ring = sR[yo & 3];
        sum = next;
        if (kWalls && (yo < 0 || yo >= g.ny)) {   // a virtual wall row
            ring[t + 1] = splat(0.0f);
            if (halo) ring[sh] = splat(0.0f);
            return;
        }
        const bool bottom = kWalls && yo == 0, top = kWalls && yo == g.ny - 1;
        C f[9];
        pull_stage<W>(st, bottom, top, k, f);
        next = sum_cells(f);
        ring[t + 1] = swap2(density_of<T>(next, shift));
        if (halo) {
            pull_stage<W>(st, bottom, top, kh, f);
            ring[sh] = swap2(density_of<T>(sum_cells(f), shift));
        }
    };
    auto collide = [&](int y, const C* st) {
        if (owner) {
            C f[9];
            pull_stage<W>(st, kWalls && y == 0, kWalls && y == g.ny - 1, k, f);
            good &= collide_cells<T, kWalls>(f, sum, ring_nbr(sR[(y - 1) & 3], sR[y & 3], sR[(y + 1) & 3], t + 1), g.ny, ph,
                                             y, site, seed, f);
#pragma unroll
            for (int i = 0; i < 9; ++i) q[(size_t)i * g.plane] = f[i];
            if (edge) {   // periodic ghost copy
                C* qg = q + (x < 2 ? g.nx : -g.nx);
#pragma unroll
                for (int i = 0; i < 9; ++i) qg[(size_t)i * g.plane] = f[i];
            }
        }
        q += g.pitch;
        site += site_row;
    };
    sweep_tile(R, densities, collide);
    if (!good) atomicOr(flag, 1);
}
template <typename T, int TW = kBlockTileW, bool kWithhold = false>
__device__ __forceinline__ void block_tile(const Cell<T>* __restrict__ fin, Cell<T>* __restrict__ fout, const Grid& g,
                                           const Physics& ph, int x0, int y0, int y1, unsigned char* dsm,
                                           BlockRingT<TW>& sR, uint32_t seed, int* flag) {
    if (kWithhold || tile_has_walls(y0, y1, g.ny))
        block_sweep<T, TW, true, kWithhold>(fin, fout, g, ph, x0, y0, y1, dsm, sR, seed, flag);
    else
        block_sweep<T, TW, false, kWithhold>(fin, fout, g, ph, x0, y0, y1, dsm, sR, seed, flag);
}

// ---------------------------------------------------------------------------
// Decoupled block tile (LBM_KERNEL_DECOUPLED).  The row stages, pulls and
// collision of block_tile without its block barrier per row: each warp keeps the
// densities of its own 32 columns, and of the two columns beside them (lanes 0 and
// 31 pull those as well), in a density ring of its own, and a stage is handed back
// through an "empty" mbarrier on which each warp arrives once it no longer reads
// the stage's row.  A warp waits only for the rows it reads (full barriers); warp
// 0, whose lanes 0-8 issue the copies, also waits until every warp has handed back
// the stage it refills.  Stage indices and barrier phases advance incrementally,
// without a division by the stage count.
// ---------------------------------------------------------------------------
template <typename T, int TW> struct DecCfg { static constexpr int kStages = 5; };
template <> struct DecCfg<__half, kWideTileW> { static constexpr int kStages = 8; };
template <> struct DecCfg<__nv_bfloat16, kWideTileW> { static constexpr int kStages = 8; };

template <typename T, int TW>
size_t dec_smem_bytes() {
    return (size_t)DecCfg<T, TW>::kStages * (9 * BlockWin<T, TW>::value * sizeof(Cell<T>) + 2 * sizeof(uint64_t));
}
template <int TW> using DecRingT = float2[TW / 32][4][34];

template <typename T, int TW>
__device__ __forceinline__ void dec_tile(const Cell<T>* __restrict__ fin, Cell<T>* __restrict__ fout, const Grid& g,
                                         const Physics& ph, int x0, int y0, int y1, unsigned char* dsm,
                                         DecRingT<TW>& sR, uint32_t seed, int* flag) {
    typedef Cell<T> C;
    constexpr int W = BlockWin<T, TW>::value, slack = BlockWin<T, TW>::kSlack;
    constexpr int S = DecCfg<T, TW>::kStages;
    constexpr int NW = TW / 32;
    C* stage = reinterpret_cast<C*>(dsm);
    uint64_t* full = reinterpret_cast<uint64_t*>(dsm + (size_t)S * 9 * W * sizeof(C));
    uint64_t* empty = full + S;
    const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
    const int rfirst = max(y0 - 2, 0);
    const int rlast = min(y1 + 1, g.ny - 1);
    const int x = x0 + t;
    const bool owner = x < g.nx;
    const int k = t + 2 + slack;
    // lanes 0 / 31 also supply the densities of the columns beside the warp
    const bool halo = lane == 0 || lane == 31;
    const int kh = lane == 0 ? k - 1 : k + 1;
    const int sh = lane == 0 ? 0 : 33;
    const C* win = fin + (g.origin + x0 - 2 - slack);
    const float2 shift = shift_of(ph);
    const uint32_t row_bytes = W * sizeof(C);
    float2(&ring)[4][34] = sR[wid];

    if (t == 0) {
        for (int j = 0; j < S; ++j) {
            mbar_init(&full[j], 1);
            mbar_init(&empty[j], NW);
        }
        mbar_fence_init();
    }
    __syncthreads();   // barriers initialised: the only block barrier

    // producer state (warp 0): the next row to issue, its stage, the phase of that
    // stage's empty barrier to wait for, and whether the stage has been used before
    int next = rfirst, nj = 0;
    uint32_t ep = 0;
    bool reuse = false;
    auto issue_next = [&]() {   // warp 0, all lanes
        if (reuse) mbar_wait(&empty[nj], ep, flag);
        const uint32_t planes = tile_row_planes(next, y0, y1, g.ny);
        if (lane == 0) mbar_expect_tx(&full[nj], (uint32_t)__popc(planes) * row_bytes);
        __syncwarp();
        if (lane < 9 && ((planes >> lane) & 1u)) {
            fence_proxy_async_smem();
            bulk_copy_g2s(stage + (size_t)nj * 9 * W + lane * W, win + (size_t)next * g.pitch + (size_t)lane * g.plane,
                          row_bytes, &full[nj]);
        }
        ++next;
        if (++nj == S) {
            nj = 0;
            if (reuse) ep ^= 1u;
            reuse = true;
        }
    };
    if (wid == 0)
        while (next <= rlast && next < rfirst + S) issue_next();

    // consumer state (every warp): rows waited for and rows handed back, in order
    int wr = rfirst, wj = 0;
    uint32_t wp = 0;
    auto wait_upto = [&](int r) {
        for (; wr <= r && wr <= rlast; ++wr) {
            mbar_wait(&full[wj], wp, flag);
            if (++wj == S) { wj = 0; wp ^= 1u; }
        }
    };
    int rel = rfirst, rj = 0;
    auto release_upto = [&](int r) {
        __syncwarp();
        for (; rel <= r && rel <= rlast; ++rel) {
            if (lane == 0) mbar_arrive(&empty[rj]);
            if (++rj == S) rj = 0;
        }
    };
    auto stage_ptr = [&](int j) -> const C* { return stage + (size_t)j * 9 * W; };
    auto wrap = [&](int j) { return j < 0 ? j + S : (j >= S ? j - S : j); };
    // pull of row yo whose own stage is jc (rows yo - 1 / yo + 1 in the stages beside it)
    auto pull_row = [&](int yo, int jc, int kk, C f[9]) {
        const C* sS = stage_ptr(wrap(jc - 1));
        const C* sC = stage_ptr(jc);
        const C* sN = stage_ptr(wrap(jc + 1));
        if (yo > 0 && yo < g.ny - 1)
            pull_cells<W>(sS, sC, sN, false, false, kk, f);
        else
            pull_cells<W>(sS, sC, sN, yo == 0, yo == g.ny - 1, kk, f);
    };
    auto densities = [&](int yo, int jc, C f[9]) -> float2 {
        pull_row(yo, jc, k, f);
        const float2 sum = sum_cells(f);
        ring[yo & 3][lane + 1] = swap2(density_of<T>(sum, shift));
        if (halo) {
            C fh[9];
            pull_row(yo, jc, kh, fh);
            ring[yo & 3][sh] = swap2(density_of<T>(sum_cells(fh), shift));
        }
        return sum;
    };
    auto zero_row = [&](int yo) {   // the virtual wall rows y = -1 and y = ny
        ring[yo & 3][lane + 1] = splat(0.0f);
        if (halo) ring[yo & 3][sh] = splat(0.0f);
    };

    // jn: stage of row y + 1 during the collision of row y (rows are consecutive from
    // rfirst, so the stage of row r is (r - rfirst) mod S)
    C fa[9], fb[9];
    float2 da, db = splat(0.0f);
    int jy = (y0 - rfirst) % S;   // stage of row y0 (a one-time division)
    if (y0 > 0) {
        wait_upto(y0);
        densities(y0 - 1, wrap(jy - 1), fb);
    } else {
        zero_row(y0 - 1);
    }
    wait_upto(y0 + 1);
    da = densities(y0, jy, fa);
    release_upto(y0 - 2);
    if (wid == 0)
        while (next <= rlast && next - S <= y0 - 2) issue_next();
    int jn = wrap(jy + 1);

    auto row = [&](int y, const C cur[9], float2 dcur, C nxt[9], float2& dnxt) {
        if (y + 1 < g.ny) {
            wait_upto(y + 2);
            dnxt = densities(y + 1, jn, nxt);
        } else {
            zero_row(y + 1);
        }
        release_upto(y - 1);   // includes the __syncwarp that publishes the ring writes
        if (wid == 0)
            while (next <= rlast && next - S <= y - 1) issue_next();
        jn = wrap(jn + 1);
        if (owner) {
            C out[9];
            if (!collide_cells<T, true>(cur, dcur, ring_nbr(ring[(y - 1) & 3], ring[y & 3], ring[(y + 1) & 3], lane + 1),
                                        g.ny, ph, y, site_index(g, y, x), seed, out))
                atomicOr(flag, 1);
            store_cells(fout, g, y, x, out);
        }
    };
    for (int y = y0; y < y1; y += 2) {
        row(y, fa, da, fb, db);
        if (y + 1 < y1) row(y + 1, fb, db, fa, da);
    }
}

template <typename T, int TW>
__global__ void __launch_bounds__(TW, 512 / TW)
step_dec_kernel(const Cell<T>* __restrict__ fin, Cell<T>* __restrict__ fout, Grid g, Physics ph, int* flag) {
    extern __shared__ __align__(128) unsigned char dsm[];
    __shared__ DecRingT<TW> sR;
    const int y0 = (int)(((long long)blockIdx.y * g.ny) / gridDim.y);
    const int y1 = (int)(((long long)(blockIdx.y + 1) * g.ny) / gridDim.y);
    const uint32_t seed = launch_seed(ph);
    advance_step(ph, blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0);
    dec_tile<T, TW>(fin, fout, g, ph, blockIdx.x * TW, y0, y1, dsm, sR, seed, flag);
}

// ---------------------------------------------------------------------------
// Paired-column block tile for 16-bit storage.  The rows, stages and pulls of
// block_tile with tiles of kWideTileW columns, but half as many threads: thread t
// owns the neighbouring columns x0 + 2t and x0 + 2t + 1.  The per-row work that does
// not depend on the site (the waits, stage addressing, the block barrier, the copy
// issue, loop control, constants) is then shared by two sites, and a column pair's
// cells are one 64-bit store per direction.  The arithmetic, and the stochastic
// rounding's random bits, are those of block_tile: the results are identical bit for
// bit.
// ---------------------------------------------------------------------------
constexpr int kPairThreads = kWideTileW / 2;
constexpr int kPairStages = 5;
// Densities as (B, A): slot 2 + c holds column x0 + c (a thread's pair 16-byte
// aligned), slots 1 and kWideTileW + 2 the halo columns.
typedef float2 PairRing[4][kWideTileW + 4];

template <typename T>
__host__ __device__ constexpr size_t pair_smem_bytes() {
    return (size_t)kPairStages * (9 * BlockWin<T, kWideTileW>::value * sizeof(Cell<T>) + sizeof(uint64_t));
}

template <typename C> __device__ __forceinline__ C cell_of_bits(uint32_t v) { return *reinterpret_cast<const C*>(&v); }
template <typename C> __device__ __forceinline__ uint32_t bits_of_cell(C v) { return *reinterpret_cast<const uint32_t*>(&v); }

template <typename T, bool kWalls>
__device__ __forceinline__ void pair_sweep(const Cell<T>* __restrict__ fin, Cell<T>* __restrict__ fout, const Grid& g,
                                           const Physics& ph, int x0, int y0, int y1, unsigned char* dsm, PairRing& sR,
                                           uint32_t seed, int* flag) {
    typedef Cell<T> C;
    constexpr int TW = kWideTileW, S = kPairStages;
    constexpr int W = BlockWin<T, TW>::value, slack = BlockWin<T, TW>::kSlack;
    static_assert(sizeof(C) == 4 && W % 2 == 0 && slack % 2 == 0, "column pairs are 8-byte aligned");
    TileRows<T, TW, S, false> R(fin, g, x0, y0, y1, dsm, flag);
    const int t = threadIdx.x;
    const int xa = x0 + 2 * t;
    const bool own_a = xa < g.nx, own_b = xa + 1 < g.nx;
    const bool edge = xa < 2 || xa + 1 >= g.nx - 2;
    const int ka = 2 * t + 2 + slack;   // window column of xa
    // threads 64 / 65: the halo columns x0 - 1 / x0 + TW
    const bool halo = t == 64 || t == 65;
    const int kh = t == 64 ? 1 + slack : TW + 2 + slack;
    const int sh = t == 64 ? 1 : TW + 2;
    const float2 shift = shift_of(ph);
    C* q = fout + (size_t)y0 * g.pitch + g.origin + xa;
    uint32_t site = site_index(g, y0, xa);
    const uint32_t site_row = site_index(g, 1, xa) - site_index(g, 0, xa);
    bool good = true;
    // sums of the stored values of rows y and y + 1
    float2 da = splat(0.0f), db = splat(0.0f), na = splat(0.0f), nb = splat(0.0f);
    // the pair's cells of row yo: directions without an x shift (and bounced-back ones)
    // are one 64-bit load
    auto pull_pair = [&](int yo, const C* st, C fa[9], C fb[9]) {
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            const C* p = st + i * W + ka;
            if (cx(i) == 0 || (kWalls && ((cy(i) == 1 && yo == 0) || (cy(i) == -1 && yo == g.ny - 1)))) {
                const uint2 v = *reinterpret_cast<const uint2*>(p);
                fa[i] = cell_of_bits<C>(v.x);
                fb[i] = cell_of_bits<C>(v.y);
            } else {
                fa[i] = p[-cx(i)];
                fb[i] = p[1 - cx(i)];
            }
        }
    };
    auto densities = [&](int yo, const C* st) {
        float2* ring = sR[yo & 3];
        da = na;
        db = nb;
        if (kWalls && (yo < 0 || yo >= g.ny)) {   // a virtual wall row
            *reinterpret_cast<float4*>(&ring[2 * t + 2]) = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            if (halo) ring[sh] = splat(0.0f);
            return;
        }
        C fa[9], fb[9];
        pull_pair(yo, st, fa, fb);
        na = sum_cells(fa);
        nb = sum_cells(fb);
        const float2 ra = density_of<T>(na, shift), rb = density_of<T>(nb, shift);
        *reinterpret_cast<float4*>(&ring[2 * t + 2]) = make_float4(ra.y, ra.x, rb.y, rb.x);
        if (halo) {
            pull_stage<W>(st, kWalls && yo == 0, kWalls && yo == g.ny - 1, kh, fa);
            ring[sh] = swap2(density_of<T>(sum_cells(fa), shift));
        }
    };
    auto collide = [&](int y, const C* st) {
        if (own_a) {
            C fa[9], fb[9];
            pull_pair(y, st, fa, fb);
            // columns xa - 1, xa, xa + 1 and xa + 2 of rows y - 1, y, y + 1
            const float2 *S0 = &sR[(y - 1) & 3][2 * t + 2], *S1 = &sR[y & 3][2 * t + 2], *S2 = &sR[(y + 1) & 3][2 * t + 2];
            const float4 ab0 = *reinterpret_cast<const float4*>(S0), ab1 = *reinterpret_cast<const float4*>(S1),
                         ab2 = *reinterpret_cast<const float4*>(S2);
            const float2 a0 = make_float2(ab0.x, ab0.y), b0 = make_float2(ab0.z, ab0.w);
            const float2 a1 = make_float2(ab1.x, ab1.y), b1 = make_float2(ab1.z, ab1.w);
            const float2 a2 = make_float2(ab2.x, ab2.y), b2 = make_float2(ab2.z, ab2.w);
            Nbr2 p;
            p.W = S1[-1]; p.E = b1;
            p.S = a0; p.SW = S0[-1]; p.SE = b0;
            p.N = a2; p.NW = S2[-1]; p.NE = b2;
            good &= collide_cells<T, kWalls>(fa, da, p, g.ny, ph, y, site, seed, fa);
            if (own_b) {
                p.W = a1; p.E = S1[2];
                p.S = b0; p.SW = a0; p.SE = S0[2];
                p.N = b2; p.NW = a2; p.NE = S2[2];
                good &= collide_cells<T, kWalls>(fb, db, p, g.ny, ph, y, site + 1, seed, fb);
#pragma unroll
                for (int i = 0; i < 9; ++i)
                    *reinterpret_cast<uint2*>(q + (size_t)i * g.plane) = make_uint2(bits_of_cell(fa[i]), bits_of_cell(fb[i]));
            } else {
#pragma unroll
                for (int i = 0; i < 9; ++i) q[(size_t)i * g.plane] = fa[i];
            }
            if (edge) {   // periodic ghost copies of the two first / last columns
#pragma unroll
                for (int b = 0; b < 2; ++b) {
                    const int x = xa + b;
                    if (x < g.nx && (x < 2 || x >= g.nx - 2)) {
                        C* qg = q + b + (x < 2 ? g.nx : -g.nx);
#pragma unroll
                        for (int i = 0; i < 9; ++i) qg[(size_t)i * g.plane] = b == 0 ? fa[i] : fb[i];
                    }
                }
            }
        }
        q += g.pitch;
        site += site_row;
    };
    sweep_tile(R, densities, collide);
    if (!good) atomicOr(flag, 1);
}
template <typename T>
__device__ __forceinline__ void pair_tile(const Cell<T>* __restrict__ fin, Cell<T>* __restrict__ fout, const Grid& g,
                                          const Physics& ph, int x0, int y0, int y1, unsigned char* dsm, PairRing& sR,
                                          uint32_t seed, int* flag) {
    if (tile_has_walls(y0, y1, g.ny)) pair_sweep<T, true>(fin, fout, g, ph, x0, y0, y1, dsm, sR, seed, flag);
    else pair_sweep<T, false>(fin, fout, g, ph, x0, y0, y1, dsm, sR, seed, flag);
}

template <typename T>
__global__ void __launch_bounds__(kPairThreads, 4)
step_pair_kernel(const Cell<T>* __restrict__ fin, Cell<T>* __restrict__ fout, Grid g, Physics ph, int* flag) {
    extern __shared__ __align__(128) unsigned char dsm[];
    __shared__ __align__(16) PairRing sR;
    const int y0 = (int)(((long long)blockIdx.y * g.ny) / gridDim.y);
    const int y1 = (int)(((long long)(blockIdx.y + 1) * g.ny) / gridDim.y);
    wait_previous_step();
    const uint32_t seed = launch_seed(ph);
    advance_step(ph, blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0);
    pair_tile<T>(fin, fout, g, ph, blockIdx.x * kWideTileW, y0, y1, dsm, sR, seed, flag);
}

// One grid: block (bx, by) of TW threads takes columns [TW bx, TW bx + TW) and the
// by-th of gridDim.y tiles of (nearly) equal height.
template <typename T, int TW>
__global__ void __launch_bounds__(TW, TileCfg<T, TW>::kBlocks)
step_block_kernel(const Cell<T>* __restrict__ fin, Cell<T>* __restrict__ fout, Grid g, Physics ph, int* flag) {
    extern __shared__ __align__(128) unsigned char dsm[];
    __shared__ BlockRingT<TW> sR;
    const int y0 = (int)(((long long)blockIdx.y * g.ny) / gridDim.y);
    const int y1 = (int)(((long long)(blockIdx.y + 1) * g.ny) / gridDim.y);
    wait_previous_step();
    const uint32_t seed = launch_seed(ph);
    advance_step(ph, blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0);
    block_tile<T, TW>(fin, fout, g, ph, blockIdx.x * TW, y0, y1, dsm, sR, seed, flag);
}

// The timeout test's kernel: step_block_kernel<float, 128> with the row copies withheld
// (block_tile's kWithhold), so that every bounded wait gives up and raises bit 2 of the
// guard.  Its output is garbage; the step counters are left alone.
__global__ void __launch_bounds__(kBlockTileW, 512 / kBlockTileW)
step_block_timeout_kernel(const float2* __restrict__ fin, float2* __restrict__ fout, Grid g, Physics ph, int* flag) {
    extern __shared__ __align__(128) unsigned char dsm[];
    __shared__ BlockRingT<kBlockTileW> sR;
    const int y0 = (int)(((long long)blockIdx.y * g.ny) / gridDim.y);
    const int y1 = (int)(((long long)(blockIdx.y + 1) * g.ny) / gridDim.y);
    block_tile<float, kBlockTileW, true>(fin, fout, g, ph, blockIdx.x * kBlockTileW, y0, y1, dsm, sR, 0u, flag);
}

// ---------------------------------------------------------------------------
// Ensemble step: one launch advances every member of one storage type by one time step.
// Block b takes tile b of the flat list that concatenates the members' tiles (members in
// order, each member's tiles row-major) and runs the tile code of the single-grid kernels
// with the member's grid and physics; no member waits for another, so uneven grids need
// no barrier.  TW 128 or 256: one column per thread; kEnsAuto: FP32 in 128-column tiles,
// 16-bit storage in paired 256-column tiles.
// ---------------------------------------------------------------------------
template <typename T, int TW> struct EnsTile {
    static constexpr bool kPaired = TW == kEnsAuto && IsShifted<T>::value;
    static constexpr int kCols = kPaired ? kWideTileW : (TW == kEnsAuto ? kBlockTileW : TW);
    static constexpr int kThreads = kPaired ? kPairThreads : kCols;
    static constexpr int kBlocks = kPaired ? 4 : TileCfg<T, kCols>::kBlocks;
};

template <typename T, int TW>
__global__ void __launch_bounds__(EnsTile<T, TW>::kThreads, EnsTile<T, TW>::kBlocks)
ensemble_step_kernel(const EnsMember* __restrict__ members, int n, int parity) {
    typedef EnsTile<T, TW> E;
    extern __shared__ __align__(128) unsigned char dsm[];
    const int tile = blockIdx.x;
    int lo = 0, hi = n - 1;   // last member whose first tile is <= tile
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (members[mid].tile_begin <= tile) lo = mid;
        else hi = mid - 1;
    }
    const EnsMember& M = members[lo];
    const int local = tile - M.tile_begin;
    const int tx = local % M.tiles_x, ty = local / M.tiles_x;
    const int y0 = (int)(((long long)ty * M.grid.ny) / M.tiles_y);
    const int y1 = (int)(((long long)(ty + 1) * M.grid.ny) / M.tiles_y);
    const Cell<T>* fin = (const Cell<T>*)M.buf[parity];
    Cell<T>* fout = (Cell<T>*)M.buf[parity ^ 1];
    Physics ph = M.phys;   // the member's counters, read / written as this parity dictates
    ph.step_in = M.step_ctr + parity;
    ph.step_out = M.step_ctr + (parity ^ 1);
    const uint32_t seed = launch_seed(ph);
    advance_step(ph, local == 0 && threadIdx.x == 0);
    if constexpr (E::kPaired) {
        __shared__ __align__(16) PairRing sR;
        pair_tile<T>(fin, fout, M.grid, ph, tx * E::kCols, y0, y1, dsm, sR, seed, M.flag);
    } else {
        __shared__ BlockRingT<E::kCols> sR;
        block_tile<T, E::kCols>(fin, fout, M.grid, ph, tx * E::kCols, y0, y1, dsm, sR, seed, M.flag);
    }
}

template <typename T, int TW>
static EnsKernel ens_kernel_of() {
    typedef EnsTile<T, TW> E;
    EnsKernel k;
    k.fn = ensemble_step_kernel<T, TW>;
    k.cols = E::kCols;
    k.threads = E::kThreads;
    if constexpr (E::kPaired) k.smem = pair_smem_bytes<T>();
    else k.smem = block_smem_bytes<T, E::kCols>();
    return k;
}
template <typename T>
static EnsKernel ens_kernel_of(int tile_x) {
    return tile_x == kWideTileW ? ens_kernel_of<T, kWideTileW>()
           : tile_x == kBlockTileW ? ens_kernel_of<T, kBlockTileW>() : ens_kernel_of<T, kEnsAuto>();
}
EnsKernel ensemble_kernel(int storage, int tile_x) {
    switch (storage) {
        case LBM_STORE_F16: return ens_kernel_of<__half>(tile_x);
        case LBM_STORE_BF16: return ens_kernel_of<__nv_bfloat16>(tile_x);
        default: return ens_kernel_of<float>(tile_x);
    }
}

// Resident blocks of an ensemble kernel on the current device (its dynamic shared memory
// allowed first).
cudaError_t ensemble_slots(const EnsKernel& k, int* slots) {
    int dev = 0, sms = 0, occ = 0;
    cudaError_t e = cudaFuncSetAttribute(k.fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)k.smem);
    if (e == cudaSuccess) e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k.fn, k.threads, k.smem);
    *slots = std::max(1, sms * occ);
    return e;
}

cudaError_t launch_ensemble_step(const EnsKernel& k, const EnsMember* d_members, int n, int tiles, int parity,
                                 cudaStream_t st) {
    (void)cudaGetLastError();
    k.fn<<<tiles, k.threads, k.smem, st>>>(d_members, n, parity);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Two-pass step: densities, as (B, A), into psi, then pull + collide reading psi
// neighbours.
// ---------------------------------------------------------------------------
template <typename T>
__global__ void __launch_bounds__(kThreadsX)
density_kernel(const Cell<T>* __restrict__ fin, float2* __restrict__ psi, Grid g, Physics ph) {
    const int x = blockIdx.x * kThreadsX + threadIdx.x;
    const int y = blockIdx.y;
    if (x >= g.nx) return;
    const int xm = x == 0 ? g.nx - 1 : x - 1;
    const int xp = x == g.nx - 1 ? 0 : x + 1;
    float2 f[9];
    pull_site<T>(fin, g, shift_of(ph), y, x, xm, xp, f);
    psi[(size_t)y * g.pitch + x] = swap2(sum9_2(f));
}

template <typename T>
__global__ void __launch_bounds__(kThreadsX)
collide_kernel(const Cell<T>* __restrict__ fin, const float2* __restrict__ psi, Cell<T>* __restrict__ fout, Grid g,
               Physics ph, int* flag) {
    const int x = blockIdx.x * kThreadsX + threadIdx.x;
    const int y = blockIdx.y;
    const uint32_t seed = launch_seed(ph);
    advance_step(ph, blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0);
    if (x >= g.nx) return;
    const int xm = x == 0 ? g.nx - 1 : x - 1;
    const int xp = x == g.nx - 1 ? 0 : x + 1;
    float2 f[9];
    pull_site<T>(fin, g, shift_of(ph), y, x, xm, xp, f);
    const float2* r = psi + (size_t)y * g.pitch;
    Nbr2 p;
    p.E = __ldg(r + xp);
    p.W = __ldg(r + xm);
    p.N = p.NE = p.NW = p.S = p.SE = p.SW = splat(0.0f);
    if (y + 1 < g.ny) {
        const float2* q = r + g.pitch;
        p.N = __ldg(q + x); p.NE = __ldg(q + xp); p.NW = __ldg(q + xm);
    }
    if (y > 0) {
        const float2* q = r - g.pitch;
        p.S = __ldg(q + x); p.SE = __ldg(q + xp); p.SW = __ldg(q + xm);
    }
    if (!collide_site<Exact<T>::value, true>(f, sum9_2(f), p, ph, y, g.ny)) atomicOr(flag, 1);
    store_step<T>(fout, g, y, x, f, shift_of(ph), seed);
}

// ---------------------------------------------------------------------------
// Initial state (Section 2, last paragraph): densities of a tanh interface at
// height y0(x), fluid at rest, f = w_i rho_s; stored as the buffer whose pull
// gives those populations.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void init_rho(const double* y0, int x, int y, double mA, double mB,
                                         double eps, double width, double& rA, double& rB) {
    const double H = 0.5 * (1.0 + tanh(((double)y - y0[x]) / width));
    rA = mA * (eps + (1.0 - eps) * H);
    rB = mB * (eps + (1.0 - eps) * (1.0 - H));
}

// y0 holds the interface heights of columns -1 .. nx (y0[x + 1]): the population a
// site sends towards x + c_i is that of the site it reaches, beside the grid too.
template <typename T>
__global__ void init_kernel(Cell<T>* __restrict__ fout, Grid g, float sA, float sB, const double* __restrict__ y0,
                            double mA, double mB, double eps, double width) {
    const int x = blockIdx.x * kThreadsX + threadIdx.x;
    const int y = blockIdx.y;
    if (x >= g.nx) return;
    const float2 shift = make_float2(sA, sB);
    double here[2];
    y0 += 1;
    init_rho(y0, x, y, mA, mB, eps, width, here[0], here[1]);
    float2 f[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        const int ty = y + cy(i);
        const int tx = x + cx(i);
        double r[2] = {here[0], here[1]};
        if (ty >= 0 && ty < g.ny) init_rho(y0, tx, ty, mA, mB, eps, width, r[0], r[1]);
        f[i] = make_float2((float)(wd(i) * r[0]), (float)(wd(i) * r[1]));
    }
    store_site<T>(fout, g, y, x, f, shift);
}

template <typename T, typename V>
__global__ void pull_to_host_kernel(const Cell<T>* __restrict__ fin, Grid g, float sA, float sB, V* __restrict__ S) {
    const int x = blockIdx.x * kThreadsX + threadIdx.x;
    const int y = blockIdx.y;
    if (x >= g.nx) return;
    // the columns beside the grid from the ghost columns (periodic copies, or a split
    // grid's neighbours)
    float2 f[9];
    pull_site<T>(fin, g, make_float2(sA, sB), y, x, x - 1, x + 1, f);
    const size_t n = (size_t)g.nx * g.ny, k = (size_t)y * g.nx + x;
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        S[(size_t)i * n + k] = (V)f[i].x;
        S[(size_t)(9 + i) * n + k] = (V)f[i].y;
    }
}

template <typename T, typename V>
__global__ void push_from_host_kernel(const V* __restrict__ S, Grid g, float sA, float sB, Cell<T>* __restrict__ fout) {
    const int x = blockIdx.x * kThreadsX + threadIdx.x;
    const int y = blockIdx.y;
    if (x >= g.nx) return;
    const size_t n = (size_t)g.nx * g.ny;
    const int xm = x == 0 ? g.nx - 1 : x - 1;
    const int xp = x == g.nx - 1 ? 0 : x + 1;
    float2 f[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        const int ty = y + cy(i);
        const int tx = cx(i) == 0 ? x : (cx(i) == 1 ? xp : xm);
        const size_t k = (ty >= 0 && ty < g.ny) ? (size_t)i * n + (size_t)ty * g.nx + tx
                                                : (size_t)opp(i) * n + (size_t)y * g.nx + x;
        f[i] = make_float2((float)S[k], (float)S[9 * n + k]);
    }
    store_site<T>(fout, g, y, x, f, make_float2(sA, sB));
}

// State files hold [component][direction][ny][pitch] planes with the ghost columns;
// column 0 sits `origin` values into a row.  V: the bits of a stored value.
template <typename V, bool kToPlanes>
__global__ void planes_kernel(V* __restrict__ cells, Grid g, V* __restrict__ planes, int pitch, int origin) {
    const int x = blockIdx.x * kThreadsX + threadIdx.x - 2;
    const int y = blockIdx.y;
    if (x >= g.nx + 2) return;
#pragma unroll
    for (int p = 0; p < 18; ++p) {
        const int s = p / 9, i = p % 9;
        V* c = cells + 2 * ((size_t)i * g.plane + (size_t)y * g.pitch + g.origin + x) + s;
        V* q = planes + ((size_t)p * g.ny + y) * pitch + origin + x;
        if (kToPlanes) *q = *c;
        else *c = *q;
    }
}

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
// Row tiles of the staged kernels: tile_y > 0 asks for at most tile_y rows per tile; 0
// makes the tiles as short as the device's resident block slots allow in one wave.  A
// launch on a small grid is a serial chain of row barriers, one per row of a tile and two
// before it, so the shortest tiles win down to one row although they read three rows for
// each they write (us per step, FP32: 128x256 24.8 with 16-row tiles, 4.0 with 1-row ones;
// 512x512 17.4 and 8.1 with 3 rows; 512x1024 19.4 and 12.6 with 5), while a second wave
// costs more than shorter tiles gain (512x256: 1 row, 1024 tiles in 912 slots 7.7, 2 rows
// 6.0).  Where one wave would make tall tiles, several waves of about kWaveRows rows: the
// blocks of an SM then are at different rows and cover each other's barriers and waits
// (10000x5000: FP16 786 us a step with one wave of 334 rows, 684 with 24 to 48 rows, 690
// with 64; FP32 1103 and 1094; 4096x4096: FP16 254 and 243, FP32 384 and 374).
constexpr int kWaveRows = 32;
int one_wave_rows(int ny, int tiles_x, int slots) {
    const int per_wave = std::max(1, slots / tiles_x);
    return (ny + per_wave - 1) / per_wave;
}
int block_tiles_y(int ny, int tiles_x, int tile_y, int slots) {
    int rows = tile_y;
    if (rows <= 0) {
        rows = one_wave_rows(ny, tiles_x, slots);
        const int waves = std::max(1, (rows + kWaveRows / 2) / kWaveRows);
        rows = (rows + waves - 1) / waves;
    }
    return (ny + rows - 1) / rows;
}

// Resident blocks of step_block_kernel<T, TW> on the current device (set up once per
// instantiation, with the kernel's dynamic shared memory attribute).
template <typename T, int TW>
static cudaError_t block_slots(int* slots) {
    static int cached = 0;
    if (cached == 0) {
        const size_t smem = block_smem_bytes<T, TW>();
        cudaError_t e = cudaFuncSetAttribute(step_block_kernel<T, TW>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)smem);
        if (e != cudaSuccess) return e;
        int dev = 0, sms = 0, occ = 0;
        if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
        if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
        if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, step_block_kernel<T, TW>, TW, smem)) !=
            cudaSuccess)
            return e;
        cached = std::max(1, sms * occ);
    }
    *slots = cached;
    return cudaSuccess;
}

// A launch that may start while the kernel before it on the stream drains (the kernels
// call wait_previous_step), where that pays.  us per step with plain and with early launches:
// launches that leave room for the next one's blocks, 128x256 FP32 3.92 and 3.49; those
// that fill the slots of 128-thread blocks, 512x1024 FP32 12.37 and 12.26, 1024x2048 FP32
// 51.3 and 50.9, 1501x999 BF16 27.7 and 27.5, and in several waves 2048x4096 FP16 126.5 and
// 126.0, 10000x5000 FP16 679 both ways.  In between, blocks that start early take the free
// slots of some SMs and leave the wave uneven (512x512 FP32, 684 blocks in 912 slots, 7.82
// and 8.24).  The 256-thread tile runs in several waves and measures the same either way
// (6000x3000 407.8 and 407.3, 10000x5000 1093.3 and 1093.0): plain.
template <typename... P, typename... A>
static cudaError_t launch_dependent(void (*kernel)(P...), dim3 grid, int threads, size_t smem, int slots, cudaStream_t st,
                                    A... args) {
    const long long blocks = (long long)grid.x * grid.y;
    const bool early = 3 * blocks <= slots || (threads == 128 && 100 * blocks >= 88LL * slots);
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &attr;
    cfg.numAttrs = early ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, P(args)...);
}

template <typename T, int TW>
static cudaError_t launch_block(const StepLaunch& L, cudaStream_t st) {
    const Grid& g = L.grid;
    int slots = 0;
    cudaError_t e = block_slots<T, TW>(&slots);
    if (e != cudaSuccess) return e;
    const int gx = (g.nx + TW - 1) / TW;
    dim3 grid(gx, block_tiles_y(g.ny, gx, L.tile_y, slots));
    return launch_dependent(step_block_kernel<T, TW>, grid, TW, block_smem_bytes<T, TW>(), slots, st, (const Cell<T>*)L.fin,
                            (Cell<T>*)L.fout, g, L.phys, L.flag);
}

// Resident blocks of step_dec_kernel<T, TW> (attribute set once per instantiation).
template <typename T, int TW>
static cudaError_t dec_slots(int* slots) {
    static int cached = 0;
    if (cached == 0) {
        const size_t smem = dec_smem_bytes<T, TW>();
        cudaError_t e = cudaFuncSetAttribute(step_dec_kernel<T, TW>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)smem);
        if (e != cudaSuccess) return e;
        int dev = 0, sms = 0, occ = 0;
        if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
        if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
        if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, step_dec_kernel<T, TW>, TW, smem)) != cudaSuccess)
            return e;
        cached = std::max(1, sms * occ);
    }
    *slots = cached;
    return cudaSuccess;
}

template <typename T, int TW>
static cudaError_t launch_dec(const StepLaunch& L, cudaStream_t st) {
    const Grid& g = L.grid;
    int slots = 0;
    cudaError_t e = dec_slots<T, TW>(&slots);
    if (e != cudaSuccess) return e;
    const int gx = (g.nx + TW - 1) / TW;
    dim3 grid(gx, block_tiles_y(g.ny, gx, L.tile_y, slots));
    step_dec_kernel<T, TW><<<grid, TW, dec_smem_bytes<T, TW>(), st>>>((const Cell<T>*)L.fin, (Cell<T>*)L.fout, g, L.phys, L.flag);
    return cudaGetLastError();
}

template <typename T>
static cudaError_t launch_pair(const StepLaunch& L, cudaStream_t st) {
    static int slots = 0;
    if (slots == 0) {
        const size_t smem = pair_smem_bytes<T>();
        cudaError_t e = cudaFuncSetAttribute(step_pair_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        int dev = 0, sms = 0, occ = 0;
        if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
        if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
        if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, step_pair_kernel<T>, kPairThreads, smem)) !=
            cudaSuccess)
            return e;
        slots = std::max(1, sms * occ);
    }
    const Grid& g = L.grid;
    const int gx = (g.nx + kWideTileW - 1) / kWideTileW;
    dim3 grid(gx, block_tiles_y(g.ny, gx, L.tile_y, slots));
    return launch_dependent(step_pair_kernel<T>, grid, kPairThreads, pair_smem_bytes<T>(), slots, st, (const Cell<T>*)L.fin,
                            (Cell<T>*)L.fout, g, L.phys, L.flag);
}

// Columns per one-column-per-thread tile: tile_x when it is 128 or 256; otherwise 256
// for 16-bit storage unless 128 span the grid, and for FP32 when the 256-column tiles hold at least kWideMinRows
// rows (tile_y, or the rows of one wave).  The wider tile reads half the halo
// columns and wins on large grids (FP32 at 10000x5000: 1094 us a step against 1103);
// tiles of 27 rows (1024x2048) run 51.4 us at 128 columns and 53.3 at 256, the barrier of 8
// warps costing more per row than the halo saves.
template <typename T>
static cudaError_t block_tile_width(const Grid& g, int tile_x, int tile_y, int* tw) {
    constexpr int kWideMinRows = 64;
    if (tile_x == kBlockTileW || tile_x == kWideTileW) {
        *tw = tile_x;
        return cudaSuccess;
    }
    if (IsShifted<T>::value) {
        *tw = g.nx > kBlockTileW ? kWideTileW : kBlockTileW;
        return cudaSuccess;
    }
    int slots = 0;
    cudaError_t e = block_slots<T, kWideTileW>(&slots);
    if (e != cudaSuccess) return e;
    const int gx = (g.nx + kWideTileW - 1) / kWideTileW;
    const int rows = tile_y > 0 ? tile_y : one_wave_rows(g.ny, gx, slots);
    *tw = rows >= kWideMinRows ? kWideTileW : kBlockTileW;
    return cudaSuccess;
}

template <typename T>
static cudaError_t launch_step_t(const StepLaunch& L, int kernel, cudaStream_t st) {
    const Grid& g = L.grid;
    (void)cudaGetLastError();   // a launch reports only its own error
    const int bx = (g.nx + kThreadsX - 1) / kThreadsX;
    if (kernel == LBM_KERNEL_TWO_PASS) {
        dim3 grid(bx, g.ny);
        density_kernel<T><<<grid, kThreadsX, 0, st>>>((const Cell<T>*)L.fin, (float2*)L.psi, g, L.phys);
        collide_kernel<T><<<grid, kThreadsX, 0, st>>>((const Cell<T>*)L.fin, (float2*)L.psi, (Cell<T>*)L.fout, g, L.phys, L.flag);
    } else if (kernel == LBM_KERNEL_STAGED || kernel == LBM_KERNEL_PAIRED) {
        // 16-bit storage at the default width: the paired-column tile (same results bit for
        // bit; FP16 at 1024x2048 36.2 us a step against 38.1 of the 256-thread tile, at
        // 10000x5000 684 against 859, at 1501x999 27.1 against 35.7), except where one
        // 128-column tile spans the grid (128x256: 4.6 us against 5.1)
        if constexpr (IsShifted<T>::value)
            if (kernel == LBM_KERNEL_PAIRED || (L.tile_x == 0 && g.nx > kBlockTileW)) return launch_pair<T>(L, st);
        int tw = 0;
        cudaError_t e = block_tile_width<T>(g, L.tile_x, L.tile_y, &tw);
        if (e != cudaSuccess) return e;
        return tw == kWideTileW ? launch_block<T, kWideTileW>(L, st) : launch_block<T, kBlockTileW>(L, st);
    } else if (kernel == LBM_KERNEL_DECOUPLED) {
        int tw = 0;
        cudaError_t e = block_tile_width<T>(g, L.tile_x, L.tile_y, &tw);
        if (e != cudaSuccess) return e;
        return tw == kWideTileW ? launch_dec<T, kWideTileW>(L, st) : launch_dec<T, kBlockTileW>(L, st);
    } else if (kernel == LBM_KERNEL_PIPE) {
        const int ty = L.tile_y > 0 ? L.tile_y : 32;
        const size_t smem = pipe_smem_bytes<T>();
        static bool attr_set = false;   // one per instantiation
        if (!attr_set) {
            cudaError_t e = cudaFuncSetAttribute(step_pipe_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                 (int)smem);
            if (e != cudaSuccess) return e;
            attr_set = true;
        }
        dim3 grid((g.nx + kPipeOwned - 1) / kPipeOwned, (g.ny + ty - 1) / ty);
        step_pipe_kernel<T><<<grid, kThreadsX, smem, st>>>((const Cell<T>*)L.fin, (Cell<T>*)L.fout, g, L.phys, ty, L.flag);
    } else if (kernel == LBM_KERNEL_WARP) {
        const int ty = L.tile_y > 0 ? L.tile_y : default_tile_y();
        const size_t smem = warp_kernel_smem_bytes<T>();
        static bool attr_set = false;   // one per instantiation
        if (!attr_set) {
            cudaError_t e = cudaFuncSetAttribute(step_warp_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                 (int)smem);
            if (e != cudaSuccess) return e;
            attr_set = true;
        }
        const int tiles_x = (g.nx + kWarpOwned - 1) / kWarpOwned;
        const int tiles = tiles_x * ((g.ny + ty - 1) / ty);
        const int blocks = (tiles + kWarpsPerBlock - 1) / kWarpsPerBlock;
        step_warp_kernel<T><<<blocks, kThreadsX, smem, st>>>((const Cell<T>*)L.fin, (Cell<T>*)L.fout, g, L.phys, ty, tiles_x,
                                                               tiles, L.flag);
    } else {
        const int ty = L.tile_y > 0 ? L.tile_y : 16;
        dim3 grid(bx, (g.ny + ty - 1) / ty);
        step_fused_kernel<T><<<grid, kThreadsX, 0, st>>>((const Cell<T>*)L.fin, (Cell<T>*)L.fout, g, L.phys, ty, L.flag);
    }
    return cudaGetLastError();
}

cudaError_t launch_step(const StepLaunch& L, int kernel, cudaStream_t st) {
    switch (L.storage) {
        case LBM_STORE_F16: return launch_step_t<__half>(L, kernel, st);
        case LBM_STORE_BF16: return launch_step_t<__nv_bfloat16>(L, kernel, st);
        default: return launch_step_t<float>(L, kernel, st);
    }
}

cudaError_t launch_step_test_timeout(const StepLaunch& L, cudaStream_t st) {
    if (L.storage != LBM_STORE_F32) return cudaErrorInvalidValue;
    (void)cudaGetLastError();
    const Grid& g = L.grid;
    const size_t smem = block_smem_bytes<float, kBlockTileW>();
    static bool attr_set = false;
    if (!attr_set) {
        cudaError_t e = cudaFuncSetAttribute(step_block_timeout_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)smem);
        if (e != cudaSuccess) return e;
        attr_set = true;
    }
    const int gx = (g.nx + kBlockTileW - 1) / kBlockTileW;
    dim3 grid(gx, std::max(1, std::min(g.ny / 8, 16)));
    step_block_timeout_kernel<<<grid, kBlockTileW, smem, st>>>((const float2*)L.fin, (float2*)L.fout, g, L.phys, L.flag);
    return cudaGetLastError();
}

cudaError_t launch_init(void* fout, const Grid& g, int storage, const float shift[2], const double* y0,
                        double mass_A, double mass_B, double minority, double width, cudaStream_t st) {
    (void)cudaGetLastError();
    dim3 grid((g.nx + kThreadsX - 1) / kThreadsX, g.ny);
    switch (storage) {
        case LBM_STORE_F16:
            init_kernel<__half><<<grid, kThreadsX, 0, st>>>((__half2*)fout, g, shift[0], shift[1], y0, mass_A, mass_B, minority, width);
            break;
        case LBM_STORE_BF16:
            init_kernel<__nv_bfloat16><<<grid, kThreadsX, 0, st>>>((__nv_bfloat162*)fout, g, shift[0], shift[1], y0, mass_A, mass_B, minority, width);
            break;
        default:
            init_kernel<float><<<grid, kThreadsX, 0, st>>>((float2*)fout, g, shift[0], shift[1], y0, mass_A, mass_B, minority, width);
    }
    return cudaGetLastError();
}

template <typename V>
static cudaError_t launch_pull_to_host(const void* fin, const Grid& g, int storage, const float shift[2], V* S,
                                       cudaStream_t st) {
    dim3 grid((g.nx + kThreadsX - 1) / kThreadsX, g.ny);
    switch (storage) {
        case LBM_STORE_F16:
            pull_to_host_kernel<__half, V><<<grid, kThreadsX, 0, st>>>((const __half2*)fin, g, shift[0], shift[1], S);
            break;
        case LBM_STORE_BF16:
            pull_to_host_kernel<__nv_bfloat16, V><<<grid, kThreadsX, 0, st>>>((const __nv_bfloat162*)fin, g, shift[0],
                                                                              shift[1], S);
            break;
        default:
            pull_to_host_kernel<float, V><<<grid, kThreadsX, 0, st>>>((const float2*)fin, g, shift[0], shift[1], S);
    }
    return cudaGetLastError();
}

template <typename V>
static cudaError_t launch_push_from_host(const V* S, const Grid& g, int storage, const float shift[2], void* fout,
                                         cudaStream_t st) {
    dim3 grid((g.nx + kThreadsX - 1) / kThreadsX, g.ny);
    switch (storage) {
        case LBM_STORE_F16:
            push_from_host_kernel<__half, V><<<grid, kThreadsX, 0, st>>>(S, g, shift[0], shift[1], (__half2*)fout);
            break;
        case LBM_STORE_BF16:
            push_from_host_kernel<__nv_bfloat16, V><<<grid, kThreadsX, 0, st>>>(S, g, shift[0], shift[1],
                                                                                (__nv_bfloat162*)fout);
            break;
        default:
            push_from_host_kernel<float, V><<<grid, kThreadsX, 0, st>>>(S, g, shift[0], shift[1], (float2*)fout);
    }
    return cudaGetLastError();
}

template <bool kToPlanes>
static cudaError_t launch_planes(void* pops, const Grid& g, int storage, void* planes, int pitch, int origin,
                                 cudaStream_t st) {
    dim3 grid((g.nx + 4 + kThreadsX - 1) / kThreadsX, g.ny);
    if (storage == LBM_STORE_F32)
        planes_kernel<uint32_t, kToPlanes><<<grid, kThreadsX, 0, st>>>((uint32_t*)pops, g, (uint32_t*)planes, pitch, origin);
    else
        planes_kernel<uint16_t, kToPlanes><<<grid, kThreadsX, 0, st>>>((uint16_t*)pops, g, (uint16_t*)planes, pitch, origin);
    return cudaGetLastError();
}
cudaError_t launch_cells_to_planes(const void* pops, const Grid& g, int storage, void* planes, int pitch, int origin,
                                   cudaStream_t st) {
    return launch_planes<true>(const_cast<void*>(pops), g, storage, planes, pitch, origin, st);
}
cudaError_t launch_planes_to_cells(const void* planes, int pitch, int origin, const Grid& g, int storage, void* pops,
                                   cudaStream_t st) {
    return launch_planes<false>(pops, g, storage, const_cast<void*>(planes), pitch, origin, st);
}

cudaError_t launch_pull_to_double(const void* fin, const Grid& g, int storage, const float shift[2], double* S,
                                  cudaStream_t st) {
    return launch_pull_to_host(fin, g, storage, shift, S, st);
}
cudaError_t launch_push_from_double(const double* S, const Grid& g, int storage, const float shift[2], void* fout,
                                    cudaStream_t st) {
    return launch_push_from_host(S, g, storage, shift, fout, st);
}
cudaError_t launch_pull_to_float(const void* fin, const Grid& g, int storage, const float shift[2], float* S,
                                 cudaStream_t st) {
    return launch_pull_to_host(fin, g, storage, shift, S, st);
}
cudaError_t launch_push_from_float(const float* S, const Grid& g, int storage, const float shift[2], void* fout,
                                   cudaStream_t st) {
    return launch_push_from_host(S, g, storage, shift, fout, st);
}

}  // namespace lbm
