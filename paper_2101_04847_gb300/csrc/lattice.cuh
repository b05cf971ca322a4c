// Device helpers shared by the kernels of liblbm: storage conversion of the
// populations and the pull of the post-streaming populations of one site.
// A buffer B holds post-collision populations in cells of both components,
// [direction][y][pitch] cells (A, B): one load brings a direction's two populations
// into a register pair, the operand of the packed FP32 instructions, and one store
// writes them (9 loads and 9 stores per site instead of 18 each; see step_kernels.cu
// for what that measured).  The post-streaming population of the kinetic equation
// (Section 2 of arXiv 2101.04847) is
//     S_i(x, y) = B_i(x - c_ix, y - c_iy)   if 0 <= y - c_iy < ny  (x periodic)
//     S_i(x, y) = B_opp(i)(x, y)            otherwise (half-way bounce-back)
#pragma once
#include "lbm_internal.cuh"

namespace lbm {

// ---------------------------------------------------------------------------
// packed FP32: two IEEE round-to-nearest operations in one instruction (FADD2 /
// FMUL2 / FFMA2).  A difference a - b is one FFMA2, b * (-1) + a, which rounds like
// the subtraction.
// ---------------------------------------------------------------------------
__device__ __forceinline__ float2 splat(float v) { return make_float2(v, v); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.0f, -1.0f), a); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 swap2(float2 a) { return make_float2(a.y, a.x); }

// ---------------------------------------------------------------------------
// storage types: float, or half / bfloat16 holding f - w_i rho0_s; a cell is the
// pair (A, B) of one direction at one site
// ---------------------------------------------------------------------------
template <typename T> struct CellOf;
template <> struct CellOf<float> { typedef float2 type; };
template <> struct CellOf<__half> { typedef __half2 type; };
template <> struct CellOf<__nv_bfloat16> { typedef __nv_bfloat162 type; };
template <typename T> using Cell = typename CellOf<T>::type;

__device__ __forceinline__ float2 to_f2(float2 v) { return v; }
__device__ __forceinline__ float2 to_f2(__half2 v) { return __half22float2(v); }
__device__ __forceinline__ float2 to_f2(__nv_bfloat162 v) { return __bfloat1622float2(v); }
// rounded to nearest even
template <typename T> __device__ __forceinline__ Cell<T> from_f2(float2 v);
template <> __device__ __forceinline__ float2 from_f2<float>(float2 v) { return v; }
template <> __device__ __forceinline__ __half2 from_f2<__half>(float2 v) { return __float22half2_rn(v); }
template <> __device__ __forceinline__ __nv_bfloat162 from_f2<__nv_bfloat16>(float2 v) { return __float22bfloat162_rn(v); }

template <typename T> struct IsShifted { static constexpr bool value = true; };
template <> struct IsShifted<float> { static constexpr bool value = false; };

// The populations (A, B) of direction i from a stored cell.
template <typename T>
__device__ __forceinline__ float2 cell_pops(Cell<T> c, int i, float2 shift) {
    const float2 v = to_f2(c);
    if constexpr (IsShifted<T>::value) return fma2(splat(wf(i)), shift, v);
    else return v;
}

// Pull the 18 post-streaming populations of column xc (neighbours xm, xp) on row y.
template <typename T>
__device__ __forceinline__ void pull_site(const Cell<T>* __restrict__ fin, const Grid& g, float2 shift, int y, int xc,
                                          int xm, int xp, float2 f[9]) {
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        const int sy = y - cy(i);
        const int sx = cx(i) == 0 ? xc : (cx(i) == 1 ? xm : xp);
        const bool inside = (cy(i) == 0) || (sy >= 0 && sy < g.ny);
        const size_t idx = inside ? (size_t)i * g.plane + (size_t)sy * g.pitch + g.origin + sx
                                  : (size_t)opp(i) * g.plane + (size_t)y * g.pitch + g.origin + xc;
        f[i] = cell_pops<T>(__ldg(fin + idx), i, shift);
    }
}

// Store the 9 cells c of column x on row y, plus the periodic ghost copy of the two
// first / last columns (read by the staged kernels' row windows).  The ghost copies
// take a separate branch, taken only by threads of edge columns.
template <typename C>
__device__ __forceinline__ void store_cells(C* __restrict__ fout, const Grid& g, int y, int x, const C c[9]) {
    C* q = fout + (size_t)y * g.pitch + g.origin + x;
#pragma unroll
    for (int i = 0; i < 9; ++i) q[(size_t)i * g.plane] = c[i];
    if (x < 2 || x >= g.nx - 2) {
        C* qg = q + (x < 2 ? g.nx : -g.nx);
#pragma unroll
        for (int i = 0; i < 9; ++i) qg[(size_t)i * g.plane] = c[i];
    }
}

// Store the 18 post-collision populations of column x on row y, rounded to nearest.
template <typename T>
__device__ __forceinline__ void store_site(Cell<T>* __restrict__ fout, const Grid& g, int y, int x, const float2 f[9],
                                           float2 shift) {
    Cell<T> c[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        float2 v = f[i];
        if constexpr (IsShifted<T>::value) v = fma2(splat(-wf(i)), shift, v);
        c[i] = from_f2<T>(v);
    }
    store_cells(fout, g, y, x, c);
}

// ---------------------------------------------------------------------------
// Stochastic rounding of the 16-bit stores.  Rounding to nearest lets slowly
// varying populations round the same way step after step, which drifts the
// masses by several per cent over 10^4 steps.  A value is instead rounded up in
// magnitude with probability equal to its distance from the lower neighbour, in
// units of the spacing: uniform random bits are added below the kept mantissa of
// the FP32 pattern and the sum is truncated.  The random bits are a hash of the
// site, the component and the time step (lowbias32 of C. Wellons' hash
// prospector; a counter-based generator, so results are reproducible), stepped
// by the PCG multiplier of M. E. O'Neill per value.  The time step matters: a
// hash of the values alone repeats its decisions in slowly varying regions and
// drifts the masses by ~1e-4 per 5000 steps.  FP16 subnormals (|h| < 2^-14) keep
// a truncation bias below 2^-24.
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t hash_lowbias32(uint32_t x) {
    x ^= x >> 16;
    x *= 0x7feb352dU;
    x ^= x >> 15;
    x *= 0x846ca68bU;
    x ^= x >> 16;
    return x;
}
// Seed of a launch's stochastic rounding: a hash of its time step (0 without a counter).
__device__ __forceinline__ uint32_t launch_seed(const Physics& ph) {
    return ph.step_in ? hash_lowbias32(*ph.step_in * 0x9E3779B9u + 0x7F4A7C15u) : 0u;
}
// The one thread `leader` of a launch passes the time step on to the next launch.
__device__ __forceinline__ void advance_step(const Physics& ph, bool leader) {
    if (leader && ph.step_out) *ph.step_out = *ph.step_in + 1u;
}

// Two FP32 values with the random bits added, truncated and packed into a cell.
template <typename T> struct SrBits;
template <> struct SrBits<__half> { static constexpr int kDrop = 13; };          // mantissa bits dropped
template <> struct SrBits<__nv_bfloat16> { static constexpr int kDrop = 16; };
__device__ __forceinline__ uint32_t pack_rz(float2 v, __half*) {
    uint32_t d;
    asm("cvt.rz.f16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(v.y), "f"(v.x));
    return d;
}
__device__ __forceinline__ uint32_t pack_rz(float2 v, __nv_bfloat16*) {
    uint32_t d;
    asm("cvt.rz.bf16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(v.y), "f"(v.x));
    return d;
}

// A site's index in the whole grid, so that a split grid draws the same bits.
__device__ __forceinline__ uint32_t site_index(const Grid& g, int y, int x) {
    return g.nx_total > 0 ? (uint32_t)y * (uint32_t)g.nx_total + (uint32_t)(g.x_offset + x)
                          : (uint32_t)y * (uint32_t)g.nx + (uint32_t)x;
}
// The 9 cells of a site from its shifted values h (16-bit storage: h is what is
// stored, no shift applied here), stochastically rounded.
template <typename T>
__device__ __forceinline__ void round_site(uint32_t site, const float2 h[9], uint32_t seed, Cell<T> c[9]) {
    constexpr int kShift = 32 - SrBits<T>::kDrop;
    uint32_t ra = hash_lowbias32((site * 2u) ^ seed), rb = hash_lowbias32((site * 2u + 1u) ^ seed);
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        ra = ra * 747796405u + 2891336453u;
        rb = rb * 747796405u + 2891336453u;
        const float2 d = make_float2(__uint_as_float(__float_as_uint(h[i].x) + (ra >> kShift)),
                                     __uint_as_float(__float_as_uint(h[i].y) + (rb >> kShift)));
        const uint32_t p = pack_rz(d, static_cast<T*>(nullptr));
        c[i] = *reinterpret_cast<const Cell<T>*>(&p);
    }
}

// Store of a time step's result f: FP32 storage as it is; 16-bit storage as
// h = f - w_i rho0_s with the stochastic rounding above.
template <typename T>
__device__ __forceinline__ void store_step(Cell<T>* __restrict__ fout, const Grid& g, int y, int x, const float2 f[9],
                                           float2 shift, uint32_t seed) {
    if constexpr (IsShifted<T>::value) {
        float2 h[9];
#pragma unroll
        for (int i = 0; i < 9; ++i) h[i] = fma2(splat(-wf(i)), shift, f[i]);
        Cell<T> c[9];
        round_site<T>(site_index(g, y, x), h, seed, c);
        store_cells(fout, g, y, x, c);
    } else {
        store_cells(fout, g, y, x, f);
    }
}

// sum of nine values, associated as ((0+1)+(2+3)) + ((4+5)+(6+7)) + 8
__device__ __forceinline__ float2 sum9_2(const float2* f) {
    const float2 lo = add2(add2(f[0], f[1]), add2(f[2], f[3]));
    const float2 hi = add2(add2(f[4], f[5]), add2(f[6], f[7]));
    return add2(add2(lo, hi), f[8]);
}

// Densities and total momentum of one site's gathered populations, summed in one
// fixed order (the mass sums and the correction must see the same values).
__device__ __forceinline__ void site_moments(const float2 f[9], float rho[2], float& jx, float& jy) {
    jx = 0.0f;
    jy = 0.0f;
#pragma unroll
    for (int s = 0; s < 2; ++s) {
        float r = 0.0f;
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            const float v = s == 0 ? f[i].x : f[i].y;
            r += v;
            jx += cx(i) * v;
            jy += cy(i) * v;
        }
        rho[s] = r;
    }
}

}  // namespace lbm
