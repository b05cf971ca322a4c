// Diagnostics of one state (Section 3 of arXiv 2101.04847): energies, the terms
// of the kinetic-energy budget, the split of the momentum-flux term into bulk
// pressure, Korteweg and tau-dependent parts, enstrophy, row means of the order
// parameter (mixing-layer width) and Cauchy-Crofton crossing counts (interface
// length).
//
// Precision.  The budget terms are centred differences of fields whose gradients
// are ~1e-5 of their values, so plain FP32 would lose most of their digits to
// cancellation; FP64, on the other hand, runs at a small fraction of the FP32
// rate on this GPU.  All per-site arithmetic is therefore double-float ("dfl":
// an unevaluated sum hi + lo of two floats, ~44 significant bits) built from the
// error-free transformations TwoSum (Knuth), Fast2Sum (Dekker) and the FMA
// product error (Ogita, Rump and Oishi, "Accurate sum and dot product", 2005).
// The moments are exact sums of the FP32 populations.  Block partials and the
// final sums are FP64, in a fixed order, so the results are deterministic.
//
// Two values are worked on at once, as the lanes of the packed FP32 instructions
// (dfl2): the two components, the two axes, or the two stresses.
//
// The diagnostics are one sweep over the populations (diag_sweep_kernel) and a reduction
// of its block partials.  The terms <u . div T> of the stresses T are taken by parts: with
// centred differences D, sum_y u(y) (D T)(y) over the averaged rows equals
// -sum_y T(y) (D u~)(y), u~ being u on those rows and 0 elsewhere (x is periodic), exactly.
// T is then needed at its own site only, contracted with velocity gradients, and no
// intermediate field is stored.
//
// The fields (densities and velocity of every site) take two passes of 32x8-thread
// blocks, each covering 32 columns x 64 rows (a thread takes 8 rows): moments_kernel
// and velocity_kernel.  Scratch (8-byte units per site): M[4] (rho_A, rho_B, jx, jy) as
// dfl, then the results at diag_fields_offset as doubles.
#include "lattice.cuh"

#include <algorithm>

namespace lbm {

namespace {

constexpr int DX = 32, DY = 8, RY = 8;   // a thread takes rows y0 + threadIdx.y + r DY, r < RY
constexpr int BY = DY * RY;               // rows per block
constexpr double kCs2 = 1.0 / 3.0;

// ---------------------------------------------------------------------------
// double-float arithmetic
// ---------------------------------------------------------------------------
struct dfl { float hi, lo; };   // value hi + lo with |lo| <= ulp(hi) / 2

__device__ __forceinline__ dfl two_sum(float a, float b) {
    const float s = a + b;
    const float bb = s - a;
    return {s, (a - (s - bb)) + (b - bb)};
}
__device__ __forceinline__ dfl fast_two_sum(float a, float b) {   // |a| >= |b| or a == 0
    const float s = a + b;
    return {s, b - (s - a)};
}
__device__ __forceinline__ dfl operator+(dfl a, dfl b) {
    dfl s = two_sum(a.hi, b.hi);
    const dfl t = two_sum(a.lo, b.lo);
    s.lo += t.hi;
    s = fast_two_sum(s.hi, s.lo);
    s.lo += t.lo;
    return fast_two_sum(s.hi, s.lo);
}
__device__ __forceinline__ dfl operator-(dfl a) { return {-a.hi, -a.lo}; }
__device__ __forceinline__ dfl operator-(dfl a, dfl b) { return a + (-b); }
__device__ __forceinline__ dfl operator*(dfl a, dfl b) {
    const float p = a.hi * b.hi;
    float e = fmaf(a.hi, b.hi, -p);
    e = fmaf(a.hi, b.lo, fmaf(a.lo, b.hi, e));
    return fast_two_sum(p, e);
}
__device__ __forceinline__ dfl operator*(dfl a, float b) {   // exact for b a power of two
    const float p = a.hi * b;
    const float e = fmaf(a.lo, b, fmaf(a.hi, b, -p));
    return fast_two_sum(p, e);
}
// a / b by one correction step of the FP32 quotient (remainder a - b q1 in dfl)
__device__ __forceinline__ dfl dfl_div(dfl a, dfl b) {
    const float q1 = a.hi / b.hi;
    const dfl r = a - b * q1;
    return fast_two_sum(q1, r.hi / b.hi);
}
__device__ __forceinline__ double to_d(dfl a) { return (double)a.hi + (double)a.lo; }
dfl dfl_of(double v) {   // host: nearest dfl of a double
    const float hi = (float)v;
    return {hi, (float)(v - (double)hi)};
}

struct DiagArgs {
    Grid g;
    int nx, ny;
    size_t n;           // nx * ny
    int r0, r1;         // averaged rows [r0, r1)
    // physics constants as dfl: G, body force, wall forces (G_wall / 6), external accelerations
    dfl G, gx, gw6[2], gext[2];
    dfl cs2, w1, w2, kappa, Gcs2, cK, floor_prod;
    dfl* M;             // [4][ny][nx]: rho_A, rho_B, jx, jy (fields)
    double* F;          // [4][ny][nx] doubles (fields)
    double* partials;   // [kDiagTerms][nblocks]
    double* rowpart;    // [ny][nbx]: row partials of phi
    double* rowpart_c;  // [ny][nbx]: row partials of the mass fraction rho_A / (rho_A + rho_B)
    int nblocks, nbx;   // blocks of the sweep in total / along x
    int mirror;         // 1: the pseudopotential beyond a wall is the wall row's (wall_mode 1)
};

__device__ __forceinline__ int row_of(int r) { return blockIdx.y * BY + threadIdx.y + r * DY; }

// a density field's value as the Shan-Chen force sees it: beyond a wall 0, or with
// the mirror the wall row's own value
__device__ __forceinline__ dfl at0(const dfl* f, const DiagArgs& a, int x, int y) {
    if (y < 0 || y >= a.ny) {
        if (!a.mirror) return dfl{0.0f, 0.0f};
        y = y < 0 ? 0 : a.ny - 1;
    }
    return f[(size_t)y * a.nx + x];
}

// Exact sum of FP32 terms: every TwoSum error is kept in lo (its own rounding is
// ~2^-48 of the largest term), normalised at the end.
struct Acc {
    float hi, lo;
    __device__ __forceinline__ void add(float v) {
        const dfl s = two_sum(hi, v);
        hi = s.hi;
        lo += s.lo;
    }
    __device__ __forceinline__ dfl value() const { return fast_two_sum(hi, lo); }
};

template <typename T>
__global__ void __launch_bounds__(DX * DY) moments_kernel(const Cell<T>* __restrict__ fin, DiagArgs a,
                                                         float sA, float sB) {
    const int x = blockIdx.x * DX + threadIdx.x;
#pragma unroll 1
    for (int r = 0; r < RY; ++r) {
        const int y = row_of(r);
        if (x >= a.nx || y >= a.ny) break;
        // the columns beside the grid from the ghost columns (periodic copies, or a
        // split grid's neighbours)
        float2 fp[9];
        pull_site<T>(fin, a.g, make_float2(sA, sB), y, x, x - 1, x + 1, fp);
        float f[2][9];
#pragma unroll
        for (int i = 0; i < 9; ++i) { f[0][i] = fp[i].x; f[1][i] = fp[i].y; }
        dfl rho[2], jx[2], jy[2];
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            Acc m = {f[s][0], 0.0f}, qx = {f[s][1], 0.0f}, qy = {f[s][2], 0.0f};
#pragma unroll
            for (int i = 1; i < 9; ++i) m.add(f[s][i]);
            qx.add(-f[s][3]); qx.add(f[s][5]); qx.add(-f[s][7]); qx.add(f[s][8]); qx.add(-f[s][6]);
            qy.add(-f[s][4]); qy.add(f[s][5]); qy.add(-f[s][7]); qy.add(f[s][6]); qy.add(-f[s][8]);
            rho[s] = m.value();
            jx[s] = qx.value();
            jy[s] = qy.value();
        }
        const size_t k = (size_t)y * a.nx + x;
        a.M[k] = rho[0];
        a.M[a.n + k] = rho[1];
        a.M[2 * a.n + k] = jx[0] + jx[1];
        a.M[3 * a.n + k] = jy[0] + jy[1];
    }
}

// sum_i w_i psi(x + c_i) c_i of a density field (the virtual wall rows as at0 gives them)
__device__ __forceinline__ void nbr_sum_d(const dfl* f, const DiagArgs& a, int x, int y, dfl& sx, dfl& sy) {
    const int xm = x == 0 ? a.nx - 1 : x - 1;
    const int xp = x == a.nx - 1 ? 0 : x + 1;
    const dfl E = at0(f, a, xp, y), W = at0(f, a, xm, y);
    const dfl N = at0(f, a, x, y + 1), S = at0(f, a, x, y - 1);
    const dfl NE = at0(f, a, xp, y + 1), NW = at0(f, a, xm, y + 1);
    const dfl SE = at0(f, a, xp, y - 1), SW = at0(f, a, xm, y - 1);
    const dfl d = NE - SW;
    sx = (E - W) * a.w1 + (d + (SE - NW)) * a.w2;
    sy = (N - S) * a.w1 + (d + (NW - SE)) * a.w2;
}

// rho_A, rho_B and the physical velocity of every site as doubles into F
__global__ void __launch_bounds__(DX * DY) velocity_kernel(DiagArgs a) {
    const int x = blockIdx.x * DX + threadIdx.x;
#pragma unroll 1
    for (int r = 0; r < RY; ++r) {
        const int y = row_of(r);
        if (x >= a.nx || y >= a.ny) break;
        const size_t k = (size_t)y * a.nx + x;
        const dfl rA = a.M[k], rB = a.M[a.n + k], jx = a.M[2 * a.n + k], jy = a.M[3 * a.n + k];
        dfl nAx, nAy, nBx, nBy;
        nbr_sum_d(a.M, a, x, y, nAx, nAy);
        nbr_sum_d(a.M + a.n, a, x, y, nBx, nBy);
        // wall force: sum_i w_i S(x + c_i) c_i = (0, -1/6) on row 0, (0, 1/6) on row ny-1
        dfl wA = {0.0f, 0.0f}, wB = {0.0f, 0.0f};
        if (y == 0) { wA = wA + a.gw6[0]; wB = wB + a.gw6[1]; }
        if (y == a.ny - 1) { wA = wA - a.gw6[0]; wB = wB - a.gw6[1]; }
        const dfl aAx = a.gx - a.G * nBx, aAy = (wA + a.gext[0]) - a.G * nBy;
        const dfl aBx = a.gx - a.G * nAx, aBy = (wB + a.gext[1]) - a.G * nAy;
        const dfl Fx = rA * aAx + rB * aBx, Fy = rA * aAy + rB * aBy;
        const dfl rho = rA + rB;
        const dfl ux = dfl_div(jx + Fx * 0.5f, rho), uy = dfl_div(jy + Fy * 0.5f, rho);
        a.F[k] = to_d(rA);
        a.F[a.n + k] = to_d(rB);
        a.F[2 * a.n + k] = to_d(ux);
        a.F[3 * a.n + k] = to_d(uy);
    }
}

// ---------------------------------------------------------------------------
// two dfl values as the lanes of packed FP32 operations
// ---------------------------------------------------------------------------
struct dfl2 { float2 hi, lo; };

__device__ __forceinline__ float2 neg2(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ dfl2 two_sum2(float2 a, float2 b) {
    const float2 s = add2(a, b);
    const float2 bb = sub2(s, a);
    return {s, add2(sub2(a, sub2(s, bb)), sub2(b, bb))};
}
__device__ __forceinline__ dfl2 two_diff2(float2 a, float2 b) {
    const float2 s = sub2(a, b);
    const float2 bb = sub2(s, a);
    return {s, sub2(sub2(a, sub2(s, bb)), add2(b, bb))};
}
__device__ __forceinline__ dfl2 fast_two_sum2(float2 a, float2 b) {
    const float2 s = add2(a, b);
    return {s, sub2(b, sub2(s, a))};
}
// Sums to within 2^-47 of |a| + |b|, the error that the operands' own low parts carry.
// (With the low parts' sum kept exact as in dfl's, the diagnostics come no closer to 64
// bits and take 295 us instead of 236 at 1024x2048.)
__device__ __forceinline__ dfl2 operator+(dfl2 a, dfl2 b) {
    const dfl2 s = two_sum2(a.hi, b.hi);
    return fast_two_sum2(s.hi, add2(s.lo, add2(a.lo, b.lo)));
}
__device__ __forceinline__ dfl2 operator-(dfl2 a, dfl2 b) {
    const dfl2 s = two_diff2(a.hi, b.hi);
    return fast_two_sum2(s.hi, add2(s.lo, sub2(a.lo, b.lo)));
}
// Product with the low parts' own product, which is never negative in a square: left out,
// sums of squares (kinetic energy, enstrophy, dissipation) are all low by some 2^-50.
__device__ __forceinline__ dfl2 operator*(dfl2 a, dfl2 b) {
    const float2 p = mul2(a.hi, b.hi);
    float2 e = fma2(a.hi, b.hi, neg2(p));
    e = fma2(a.hi, b.lo, fma2(a.lo, b.hi, fma2(a.lo, b.lo, e)));
    return fast_two_sum2(p, e);
}
__device__ __forceinline__ dfl2 times(dfl2 a, float2 b) {
    const float2 p = mul2(a.hi, b);
    return fast_two_sum2(p, fma2(a.lo, b, fma2(a.hi, b, neg2(p))));
}
__device__ __forceinline__ dfl2 scaled(dfl2 a, float b) { return {mul2(a.hi, splat(b)), mul2(a.lo, splat(b))}; }   // b a power of two
__device__ __forceinline__ dfl2 both(dfl a) { return {splat(a.hi), splat(a.lo)}; }
__device__ __forceinline__ dfl2 pair(dfl a, dfl b) { return {make_float2(a.hi, b.hi), make_float2(a.lo, b.lo)}; }
__device__ __forceinline__ dfl first(dfl2 a) { return {a.hi.x, a.lo.x}; }
__device__ __forceinline__ dfl second(dfl2 a) { return {a.hi.y, a.lo.y}; }
__device__ __forceinline__ dfl2 swapped(dfl2 a) { return {swap2(a.hi), swap2(a.lo)}; }
// the lanes' first values of a and b, and their second values: a transpose
__device__ __forceinline__ dfl2 firsts(dfl2 a, dfl2 b) { return pair(first(a), first(b)); }
__device__ __forceinline__ dfl2 seconds(dfl2 a, dfl2 b) { return pair(second(a), second(b)); }
__device__ __forceinline__ float2 div2(float2 a, float2 b) { return make_float2(a.x / b.x, a.y / b.y); }
// a / b by one correction step of the FP32 quotient, as dfl_div.  (Products with a rounded
// 1 / b.hi save 12 us at 1024x2048 and put 1.6 times the error into the velocity.)
__device__ __forceinline__ dfl2 quotient(dfl2 a, dfl2 b) {
    const float2 q = div2(a.hi, b.hi);
    const dfl2 r = a - times(b, q);
    return fast_two_sum2(q, div2(r.hi, b.hi));
}
// Sums: of FP32 terms exactly, as Acc (the TwoSum errors in lo), or of dfl terms.
struct Acc2 {
    float2 hi = {0.0f, 0.0f}, lo = {0.0f, 0.0f};
    __device__ __forceinline__ void add(float2 v) {
        const dfl2 s = two_sum2(hi, v);
        hi = s.hi;
        lo = add2(lo, s.lo);
    }
    __device__ __forceinline__ void add(dfl2 v) {
        const dfl2 s = dfl2{hi, lo} + v;
        hi = s.hi;
        lo = s.lo;
    }
    __device__ __forceinline__ dfl2 value() const { return fast_two_sum2(hi, lo); }
};

// ---------------------------------------------------------------------------
// The diagnostics sweep.  A block of kSweepT threads owns kSweepCols columns and the
// by-th of gridDim.y tiles of rows, swept bottom up; thread t handles column
// x0 + t - 2, the two outermost on each side only for their neighbours.  Each iteration
// takes the moments of row m (from the stored populations), the velocity of row m - 1 and
// the terms of row m - 2; densities and velocities are exchanged through rings in shared
// memory.  Row sums of phi and the mass fraction are taken kRowBatch rows at a time, 16
// threads to a row: 8 columns each in double-float, then FP64.
//
// Bound by issue: about 1.7 k mostly packed FP32 instructions per site against 72 bytes
// read.  The four passes it replaces stored 15 dfl per site, read them again with their
// neighbours and worked one value at a time: a call took 449 us at 1024x2048, 236 now, and
// no term is further from 64 bits than theirs (rms over 66 flows, relative: kinetic energy
// 2.0e-15 before and 1.2e-15 now, dissipation 2.1e-15 and 1.7e-15).
// ---------------------------------------------------------------------------
constexpr int kSweepT = 128, kSweepCols = kSweepT - 4;
constexpr int kRowBatch = 8;

struct SweepShared {
    float4 rho[8][kSweepT];            // (A.hi, B.hi, A.lo, B.lo) of row r in slot r & 7
    float4 u[4][kSweepT];              // (ux.hi, uy.hi, ux.lo, uy.lo) of row r in slot r & 3
    float4 rows[kRowBatch][kSweepT];   // (phi.hi, c.hi, phi.lo, c.lo) of the batch's rows
    double sums[kDiagTerms][kSweepT / 32];
};
__device__ __forceinline__ dfl2 dfl2_of(float4 v) { return {make_float2(v.x, v.y), make_float2(v.z, v.w)}; }
__device__ __forceinline__ float4 float4_of(dfl2 v) { return make_float4(v.hi.x, v.hi.y, v.lo.x, v.lo.y); }
// sign of rho_A - rho_B, exact for normalised values
__device__ __forceinline__ bool phi_positive(float4 r) { return r.x > r.y || (r.x == r.y && r.z > r.w); }

template <typename T>
__global__ void __launch_bounds__(kSweepT, 4)
diag_sweep_kernel(const Cell<T>* __restrict__ fin, DiagArgs a, float2 shift) {
    __shared__ SweepShared sm;
    const int t = threadIdx.x;
    const int x = blockIdx.x * kSweepCols + t - 2;
    const int xw = (x + a.nx) % a.nx;   // periodic; columns past nx + 1 only feed threads that own none
    const bool own = t >= 2 && t < kSweepT - 2 && x < a.nx;
    const int ty0 = (int)(((long long)blockIdx.y * a.ny) / gridDim.y);
    const int ty1 = (int)(((long long)(blockIdx.y + 1) * a.ny) / gridDim.y);
    const int r0 = a.r0, r1 = a.r1;

    Acc2 mass, ek_visc, om_by, ep_rho, fk_ft, iso_pb;
    int n0 = 0, n90 = 0, n45 = 0, n135 = 0;
    const dfl2 zero = {splat(0.0f), splat(0.0f)};
    dfl2 j = zero;   // momentum of the row whose velocity is next
    Cell<T> c[9];    // row m's cells, loaded one iteration ahead
    auto load = [&](int m) {
        if (m < 0 || m >= a.ny) return;
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            const int sy = m - cy(i);
            const bool inside = sy >= 0 && sy < a.ny;
            c[i] = __ldg(fin + (inside ? (size_t)i * a.g.plane + (size_t)sy * a.g.pitch + a.g.origin + (xw - cx(i))
                                       : (size_t)opp(i) * a.g.plane + (size_t)m * a.g.pitch + a.g.origin + xw));
        }
    };
    load(ty0 - 2);
    int batched = 0;   // rows in sm.rows, the last of them row `last`
    auto flush_rows = [&](int last) {
        __syncthreads();
        const int r = t >> 4, l = t & 15;
        if (r < batched) {   // whole groups of 16 lanes
            dfl2 v = dfl2_of(sm.rows[r][l]);
#pragma unroll 1
            for (int k = 1; k < kSweepT / 16; ++k) v = v + dfl2_of(sm.rows[r][l + 16 * k]);
            const unsigned mask = (t & 16) ? 0xffff0000u : 0x0000ffffu;
            double phi = to_d(first(v)), c = to_d(second(v));   // 8 columns' sums; FP64 from here on
#pragma unroll
            for (int o = 8; o > 0; o >>= 1) {
                phi += __shfl_down_sync(mask, phi, o, 16);
                c += __shfl_down_sync(mask, c, o, 16);
            }
            if (l == 0) {
                const size_t k = (size_t)(last - batched + 1 + r) * a.nbx + blockIdx.x;
                a.rowpart[k] = phi;
                a.rowpart_c[k] = c;
            }
        }
        batched = 0;
        __syncthreads();
    };

#pragma unroll 1
    for (int m = ty0 - 2; m < ty1 + 2; ++m) {
        // --- moments of row m
        const dfl2 jm = j;   // momentum of row m - 1
        if (m >= 0 && m < a.ny) {
            float2 f[9];
#pragma unroll
            for (int i = 0; i < 9; ++i) f[i] = cell_pops<T>(c[i], i, shift);
            load(m + 1);
            Acc2 r, qx, qy;
            r.hi = f[0];
            qx.hi = f[1];
            qy.hi = f[2];
#pragma unroll
            for (int i = 1; i < 9; ++i) r.add(f[i]);
            qx.add(neg2(f[3])); qx.add(f[5]); qx.add(neg2(f[7])); qx.add(f[8]); qx.add(neg2(f[6]));
            qy.add(neg2(f[4])); qy.add(f[5]); qy.add(neg2(f[7])); qy.add(f[6]); qy.add(neg2(f[8]));
            const dfl2 rho = r.value(), jx = qx.value(), jy = qy.value();
            sm.rho[m & 7][t] = float4_of(rho);
            j = firsts(jx, jy) + seconds(jx, jy);
            if (own && m >= ty0 && m < ty1) mass.add(rho);
        } else {
            load(m + 1);
        }
        __syncthreads();
        // --- velocity of row m - 1 (interior rows only: crop >= 3)
        const int yu = m - 1;
        if (yu >= r0 - 2 && yu < r1 + 2 && yu > ty0 - 2 && t >= 1 && t < kSweepT - 1) {
            const float4 *rS = &sm.rho[(yu - 1) & 7][t], *rC = &sm.rho[yu & 7][t], *rN = &sm.rho[(yu + 1) & 7][t];
            const dfl2 d = dfl2_of(rN[1]) - dfl2_of(rS[-1]), e = dfl2_of(rS[1]) - dfl2_of(rN[-1]);
            const dfl2 ew = dfl2_of(rC[1]) - dfl2_of(rC[-1]), ns = dfl2_of(rN[0]) - dfl2_of(rS[0]);
            // sum_i w_i psi(x + c_i) c_i of both components: (4 (E - W) + (NE - SW) + (SE - NW)) / 36, ...
            const dfl2 w2 = both(a.w2);
            const dfl2 sx = (scaled(ew, 4.0f) + (d + e)) * w2, sy = (scaled(ns, 4.0f) + (d - e)) * w2;
            const dfl2 rc = dfl2_of(rC[0]), G = both(a.G);
            const dfl2 ax = both(a.gx) - G * swapped(sx), ay = pair(a.gext[0], a.gext[1]) - G * swapped(sy);
            const dfl2 Fx = rc * ax, Fy = rc * ay;
            const dfl2 F = firsts(Fx, Fy) + seconds(Fx, Fy);
            const dfl2 rho = rc + swapped(rc);
            sm.u[yu & 3][t] = float4_of(quotient(jm + scaled(F, 0.5f), rho));
        }
        __syncthreads();
        // --- terms of row m - 2
        const int y = m - 2;
        if (y < ty0 || y < r0 - 1 || y > r1) continue;
        const bool avg = y >= r0 && y < r1;
        if (own) {
            const float4 *rS = &sm.rho[(y - 1) & 7][t], *rC = &sm.rho[y & 7][t], *rN = &sm.rho[(y + 1) & 7][t];
            const float4 *uS = &sm.u[(y - 1) & 3][t], *uC = &sm.u[y & 3][t], *uN = &sm.u[(y + 1) & 3][t];
            const dfl2 r = dfl2_of(rC[0]);
            // twice the density gradients of (A, B), then of phi, and the Laplacian of phi
            const dfl2 E = dfl2_of(rC[1]), Wt = dfl2_of(rC[-1]), N = dfl2_of(rN[0]), S = dfl2_of(rS[0]);
            const dfl2 gx = E - Wt, gy = N - S;
            const dfl2 P = firsts(gx, gy) - seconds(gx, gy);   // 2 (px, py)
            const dfl2 ew = E + Wt, ns = N + S;
            const dfl2 lap2 = (ew + ns) - scaled(r, 4.0f);
            // rho, phi
            const dfl2 rA = both(first(r)), rB = {make_float2(r.hi.y, -r.hi.y), make_float2(r.lo.y, -r.lo.y)};
            const dfl2 rp = rA + rB;
            const dfl rho = first(rp), phi = second(rp);
            // 2 v, v = rho_B grad rho_A - rho_A grad rho_B
            const dfl2 rs = swapped(r);
            const dfl2 cxv = rs * gx, cyv = rs * gy;
            const dfl2 V = firsts(cxv, cyv) - seconds(cxv, cyv);
            // twice the velocity gradients, and those of u~ (u on the averaged rows, else 0)
            const dfl2 dxu = dfl2_of(uC[1]) - dfl2_of(uC[-1]);   // 2 (dx ux, dx uy)
            const dfl2 dyu = dfl2_of(uN[0]) - dfl2_of(uS[0]);    // 2 (dy ux, dy uy)
            dfl2 mx = dxu, my = dyu;
            if (y <= r0 || y >= r1 - 1) {   // a row beside an edge of the averaged rows (uniform)
                if (!avg) mx = zero;
                const bool inN = y + 1 >= r0 && y + 1 < r1, inS = y - 1 >= r0 && y - 1 < r1;
                my = (inN ? dfl2_of(uN[0]) : zero) - (inS ? dfl2_of(uS[0]) : zero);
            }
            // the divergence (A + D) and the shear of u~, doubled; the shear and the curl of u
            const dfl A = first(mx), D = second(my);
            const dfl2 trsh = pair(A, second(mx)) + pair(D, first(my));
            const dfl2 curl = both(second(dxu)) +
                              dfl2{make_float2(dyu.hi.x, -dyu.hi.x), make_float2(dyu.lo.x, -dyu.lo.x)};
            const dfl2 tr = both(first(trsh)), A2 = both(A), D2 = both(D);
            // q = X^2 A + X Y S + Y^2 D for (X, Y) = 2 grad phi and 2 v
            const dfl2 X = firsts(P, V), Y = seconds(P, V);
            const dfl2 q = X * (X * A2 + Y * both(second(trsh))) + Y * Y * D2;
            // (lap phi, |2 grad phi|^2); rho_A rho_B and phi lap phi
            const dfl2 PP = P * P;
            const dfl2 ls = pair(first(lap2), first(PP)) +
                            dfl2{make_float2(-lap2.hi.y, PP.hi.y), make_float2(-lap2.lo.y, PP.lo.y)};
            const dfl2 pr = pair(first(r), phi) * pair(second(r), first(ls));
            const dfl prod = first(pr);
            dfl low = prod;
            if (low.hi < a.floor_prod.hi || (low.hi == a.floor_prod.hi && low.lo < a.floor_prod.lo)) low = a.floor_prod;
            // mass fraction and the tau stress's coefficient
            const dfl lr = low * rho;
            const dfl2 cq = quotient(pair(first(r), a.cK), pair(rho, lr));
            // isotropic part of P^K over -kappa, times (A + D): kept times 2
            const dfl ip = second(pr) + dfl{0.125f * ls.hi.y, 0.125f * ls.lo.y};
            iso_pb.add(pair(ip * first(trsh), dfl{0.0f, 0.0f}));
            // the other contractions with grad u~, kept times 8
            fk_ft.add(q * pair(a.kappa, second(cq)));
            // |u|^2; the contraction of the true gradients' normal parts with those of u~
            const dfl2 uc = avg ? dfl2_of(uC[0]) : zero;
            const dfl2 uu = uc * uc;
            const dfl2 dd = pair(first(dxu), second(dyu)) * pair(A, D);
            const dfl2 un = firsts(uu, dd) + seconds(uu, dd);
            // rho |u|^2 and the viscous contraction, kept times 4
            const dfl2 es = pair(rho, first(curl)) * pair(first(un), second(trsh));
            ek_visc.add(es);
            ek_visc.add(dfl2{make_float2(0.0f, 2.0f * un.hi.y), make_float2(0.0f, 2.0f * un.lo.y)});
            if (avg) {
                // u . grad p_b, p_b = cs2 rho + G cs2 rho_A rho_B, kept times 2: the difference of
                // the products is (gA sB + gB sA) / 2 with the neighbours' differences g and sums s
                const dfl2 mx2 = gx * swapped(ew), my2 = gy * swapped(ns);
                const dfl2 gp = (firsts(gx, gy) + seconds(gx, gy)) * both(a.cs2) +
                                (firsts(mx2, my2) + seconds(mx2, my2)) * scaled(both(a.Gcs2), 0.5f);
                const dfl2 up = uc * gp;
                iso_pb.add(dfl2{make_float2(0.0f, up.hi.x), make_float2(0.0f, up.lo.x)});
                iso_pb.add(dfl2{make_float2(0.0f, up.hi.y), make_float2(0.0f, up.lo.y)});
                const dfl om = second(curl);
                om_by.add(pair(om, second(uc)) * pair(om, phi));
                ep_rho.add(times(pair(phi, rho), make_float2((float)y, 1.0f)));
                // crossing counts of (phi > 0) for pairs starting at (x, y)
                const bool p = phi_positive(rC[0]);
                n0 += p != phi_positive(rC[1]);
                if (y + 1 < r1) {
                    n90 += p != phi_positive(rN[0]);
                    n45 += p != phi_positive(rN[1]);
                    n135 += p != phi_positive(rN[-1]);
                }
                const dfl cA = rho.hi > 0.0f ? first(cq) : dfl{0.0f, 0.0f};
                sm.rows[batched][t] = make_float4(phi.hi, cA.hi, phi.lo, cA.lo);
            }
        } else if (avg) {
            sm.rows[batched][t] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        }
        if (avg && (++batched == kRowBatch || y == r1 - 1 || y == ty1 - 1)) flush_rows(y);
    }

    // block sums of the terms, FP64 from here on; the powers of two that the doubled
    // gradients left, and the sign of the summation by parts, are taken off
    const int lane = t & 31, warp = t >> 5;
    const dfl2 iso = iso_pb.value();
    const double kappa = to_d(a.kappa);
    const dfl2 v[5] = {mass.value(), ek_visc.value(), om_by.value(), ep_rho.value(), fk_ft.value()};
    const int term[10] = {T_MASS_A, T_MASS_B, T_EK, T_VISC, T_OMEGA2, T_BUOY, T_EP, T_RHO, T_FLUX_K, T_FLUX_TAU};
    const double scale[10] = {1.0, 1.0, 0.5, -0.25, 0.25, 1.0, 1.0, 1.0, -0.125, -0.125};
    auto warp_total = [&](double d, int k) {
        for (int o = 16; o > 0; o >>= 1) d += __shfl_down_sync(0xffffffffu, d, o);
        if (lane == 0) sm.sums[k][warp] = d;
    };
#pragma unroll
    for (int k = 0; k < 10; ++k) {
        double d = scale[k] * to_d(k & 1 ? second(v[k / 2]) : first(v[k / 2]));
        if (term[k] == T_FLUX_K) d += 0.5 * kappa * to_d(first(iso));   // the isotropic part
        warp_total(d, term[k]);
    }
    warp_total(0.5 * to_d(second(iso)), T_FLUX_PB);
    warp_total((double)n0, T_N0);
    warp_total((double)n90, T_N90);
    warp_total((double)n45, T_N45);
    warp_total((double)n135, T_N135);
    __syncthreads();
    if (t < kDiagTerms) {
        double d = 0.0;
        for (int w = 0; w < kSweepT / 32; ++w) d += sm.sums[t][w];
        a.partials[(size_t)t * a.nblocks + blockIdx.y * gridDim.x + blockIdx.x] = d;
    }
}

// blocks [0, kDiagTerms): term sums over the block partials; the next blocks, a warp to
// each of the 2 (r1 - r0) rows: row sums of phi, then of the mass fraction.
__global__ void __launch_bounds__(256) reduce_kernel(DiagArgs a, double* out) {
    __shared__ double sm[8];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int nrows = a.r1 - a.r0;
    const int k = (blockIdx.x - kDiagTerms) * 8 + warp;   // row
    double s = 0.0;
    if (blockIdx.x < kDiagTerms) {
        const double* p = a.partials + (size_t)blockIdx.x * a.nblocks;
        for (int b = tid; b < a.nblocks; b += 256) s += p[b];
    } else if (k < 2 * nrows) {
        const int y = a.r0 + (k < nrows ? k : k - nrows);
        const double* p = (k < nrows ? a.rowpart : a.rowpart_c) + (size_t)y * a.nbx;
        for (int b = lane; b < a.nbx; b += 32) s += p[b];
    }
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if (blockIdx.x >= kDiagTerms) {
        if (lane == 0 && k < 2 * nrows) out[kDiagTerms + k] = s;
        return;
    }
    if (lane == 0) sm[warp] = s;
    __syncthreads();
    if (tid == 0) {
        double v = 0.0;
        for (int w = 0; w < 8; ++w) v += sm[w];
        out[blockIdx.x] = v;
    }
}

// Row tiles of the sweep on an nx x ny grid: about kSweepRows rows each, fewer where that
// leaves block slots empty.
constexpr int kSweepRows = 32, kSweepMinRows = 4, kSweepSlots = 600;
int sweep_tiles_x(int nx) { return (nx + kSweepCols - 1) / kSweepCols; }
int sweep_tiles_y(int nx, int ny) {
    const int per_wave = std::max(1, kSweepSlots / sweep_tiles_x(nx));
    const int rows = std::min(kSweepRows, std::max(kSweepMinRows, (ny + per_wave - 1) / per_wave));
    return (ny + rows - 1) / rows;
}

DiagArgs make_args(const DiagLaunch& D) {
    DiagArgs a;
    a.g = D.grid;
    a.nx = D.grid.nx;
    a.ny = D.grid.ny;
    a.n = (size_t)a.nx * a.ny;
    a.r0 = D.crop;
    a.r1 = a.ny - D.crop;
    a.G = dfl_of(D.G);
    a.gx = dfl_of(D.gx);
    a.gw6[0] = dfl_of(D.G_wall[0] / 6.0);
    a.gw6[1] = dfl_of(D.G_wall[1] / 6.0);
    a.gext[0] = dfl_of(D.g_ext[0]);
    a.gext[1] = dfl_of(D.g_ext[1]);
    a.cs2 = dfl_of(kCs2);
    a.w1 = dfl_of(1.0 / 9.0);
    a.w2 = dfl_of(1.0 / 36.0);
    a.kappa = dfl_of(kCs2 * kCs2 * D.G / 4.0);
    a.Gcs2 = dfl_of(D.G * kCs2);
    const double tm = D.tau_bar - 0.5;
    a.cK = dfl_of(kCs2 * kCs2 * tm * tm);
    a.floor_prod = dfl_of(1e-12);
    a.mirror = D.wall_mirror;
    a.M = reinterpret_cast<dfl*>(D.scratch);
    a.F = D.scratch + diag_fields_offset(a.nx, a.ny);
    a.nbx = sweep_tiles_x(a.nx);
    a.nblocks = a.nbx * sweep_tiles_y(a.nx, a.ny);
    a.partials = D.partials;
    a.rowpart = D.partials + (size_t)kDiagTerms * a.nblocks;
    a.rowpart_c = a.rowpart + (size_t)a.ny * a.nbx;
    return a;
}

template <typename T>
cudaError_t launch_moments(const DiagLaunch& D, const DiagArgs& a, cudaStream_t st) {
    dim3 grid((a.nx + DX - 1) / DX, (a.ny + BY - 1) / BY), block(DX, DY);
    moments_kernel<T><<<grid, block, 0, st>>>((const Cell<T>*)D.fin, a, D.shift[0], D.shift[1]);
    return cudaGetLastError();
}

cudaError_t moments(const DiagLaunch& D, const DiagArgs& a, cudaStream_t st) {
    switch (D.storage) {
        case LBM_STORE_F16: return launch_moments<__half>(D, a, st);
        case LBM_STORE_BF16: return launch_moments<__nv_bfloat16>(D, a, st);
        default: return launch_moments<float>(D, a, st);
    }
}

// ---------------------------------------------------------------------------
// closure network input
// ---------------------------------------------------------------------------
struct FeatArgs {
    Grid g;
    float G, gx, gw6[2], gext[2];
    float mean[4], scale[4];
    int mirror;
};

// One sweep: a block of 128 threads owns kFeatCols columns and the by-th of gridDim.y tiles
// of rows, thread t column x0 + t - 1 (the two outermost for their neighbours), with the
// densities of three rows in a ring in shared memory.  The force and physical velocity are
// those of the diagnostics, in FP32.  Bound by HBM: 72 bytes read and 24 written per site.
// A moments pass, a pass over their neighbours and one that packed the planes took 69 us at
// 1024x2048, 39 now.
constexpr int kFeatT = 128, kFeatCols = kFeatT - 2, kFeatRows = 16;

__global__ void __launch_bounds__(kFeatT) closure_input_kernel(const float2* __restrict__ fin, FeatArgs a,
                                                               float* __restrict__ rho2, uint4* __restrict__ xin,
                                                               int pitch) {
    __shared__ float2 sR[4][kFeatT];
    const int t = threadIdx.x, nx = a.g.nx, ny = a.g.ny;
    const int x = blockIdx.x * kFeatCols + t - 1;
    const int xw = (x + nx) % nx, xm = xw == 0 ? nx - 1 : xw - 1, xp = xw == nx - 1 ? 0 : xw + 1;
    const bool own = t >= 1 && t < kFeatT - 1 && x < nx;
    const int y0 = blockIdx.y * kFeatRows, y1 = min(y0 + kFeatRows, ny);
    const size_t n = (size_t)nx * ny;
    float2 f[9], j = splat(0.0f), jn = splat(0.0f);   // momenta of the row whose input is next, and of row m
    float2 r = splat(0.0f), rn = splat(0.0f);         // densities likewise
    auto load = [&](int m) {
        if (m >= 0 && m < ny) pull_site<float>(fin, a.g, splat(0.0f), m, xw, xm, xp, f);
    };
    load(y0 - 1);
#pragma unroll 1
    for (int m = y0 - 1; m <= y1; ++m) {
        j = jn;
        r = rn;
        if (m >= 0 && m < ny) {
            float rho[2], jx, jy;
            site_moments(f, rho, jx, jy);
            jn = make_float2(jx, jy);
            rn = make_float2(rho[0], rho[1]);
            sR[m & 3][t] = rn;
            if (own && m >= y0 && m < y1) {
                const size_t k = (size_t)m * nx + x;
                rho2[k] = rho[0];
                rho2[n + k] = rho[1];
            }
        }
        load(m + 1);
        __syncthreads();
        const int y = m - 1;
        if (y < y0 || !own) continue;
        // neighbours' densities, zero beyond the walls (or the wall rows' with the mirror)
        auto at = [&](int yy, int dx) {
            if (yy < 0 || yy >= ny) {
                if (!a.mirror) return splat(0.0f);
                yy = y;
            }
            return sR[yy & 3][t + dx];
        };
        const float2 E = at(y, 1), W = at(y, -1), N = at(y + 1, 0), S = at(y - 1, 0);
        const float2 d = sub2(at(y + 1, 1), at(y - 1, -1)), SE = at(y - 1, 1), NW = at(y + 1, -1);
        const float2 sx = fma2(sub2(E, W), splat(1.0f / 9.0f), mul2(add2(d, sub2(SE, NW)), splat(1.0f / 36.0f)));
        const float2 sy = fma2(sub2(N, S), splat(1.0f / 9.0f), mul2(add2(d, sub2(NW, SE)), splat(1.0f / 36.0f)));
        float wA = 0.0f, wB = 0.0f;
        if (y == 0) { wA += a.gw6[0]; wB += a.gw6[1]; }
        if (y == ny - 1) { wA -= a.gw6[0]; wB -= a.gw6[1]; }
        // each component feels the other's neighbours
        const float aAx = a.gx - a.G * sx.y, aAy = (wA + a.gext[0]) - a.G * sy.y;
        const float aBx = a.gx - a.G * sx.x, aBy = (wB + a.gext[1]) - a.G * sy.x;
        const float Fx = r.x * aAx + r.y * aBx, Fy = r.x * aAy + r.y * aBy;
        const float rho = r.x + r.y;
        const float v[4] = {r.x, r.y, (j.x + 0.5f * Fx) / rho, (j.y + 0.5f * Fy) / rho};
        float q[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) q[c] = (v[c] - a.mean[c]) / a.scale[c];
        const __nv_bfloat162 lo = __floats2bfloat162_rn(q[0], q[1]), hi = __floats2bfloat162_rn(q[2], q[3]);
        const uint4 cell = make_uint4(*reinterpret_cast<const uint32_t*>(&lo), *reinterpret_cast<const uint32_t*>(&hi), 0u, 0u);
        uint4* row = xin + (size_t)(y + 1) * pitch;
        row[x + 1] = cell;
        if (x == 0) row[nx + 1] = cell;
        if (x == nx - 1) row[0] = cell;
    }
}

}  // namespace

cudaError_t launch_closure_input(const DiagLaunch& D, float* rho2, const float mean[4], const float scale[4],
                                 uint8_t* xin, int pitch, cudaStream_t st) {
    FeatArgs a;
    a.g = D.grid;
    a.G = (float)D.G;
    a.gx = (float)D.gx;
    a.mirror = D.wall_mirror;
    for (int s = 0; s < 2; ++s) {
        a.gw6[s] = (float)(D.G_wall[s] / 6.0);
        a.gext[s] = (float)D.g_ext[s];
    }
    for (int c = 0; c < 4; ++c) {
        a.mean[c] = mean[c];
        a.scale[c] = scale[c];
    }
    const dim3 grid((D.grid.nx + kFeatCols - 1) / kFeatCols, (D.grid.ny + kFeatRows - 1) / kFeatRows);
    closure_input_kernel<<<grid, kFeatT, 0, st>>>((const float2*)D.fin, a, rho2, reinterpret_cast<uint4*>(xin), pitch);
    return cudaGetLastError();
}

size_t diag_scratch_doubles(int nx, int ny) { return diag_fields_offset(nx, ny) + (size_t)4 * nx * ny; }

size_t diag_partials_doubles(int nx, int ny) {
    const size_t gx = sweep_tiles_x(nx), gy = sweep_tiles_y(nx, ny);
    return (size_t)kDiagTerms * gx * gy + (size_t)2 * ny * gx;
}

size_t diag_fields_offset(int nx, int ny) { return (size_t)6 * nx * ny; }

template <typename T>
static cudaError_t launch_sweep(const DiagLaunch& D, const DiagArgs& a, cudaStream_t st) {
    const dim3 grid(a.nbx, a.nblocks / a.nbx);
    diag_sweep_kernel<T><<<grid, kSweepT, 0, st>>>((const Cell<T>*)D.fin, a, make_float2(D.shift[0], D.shift[1]));
    return cudaGetLastError();
}

cudaError_t launch_diagnostics(const DiagLaunch& D, cudaStream_t st) {
    (void)cudaGetLastError();   // a launch reports only its own error
    const DiagArgs a = make_args(D);
    // u is needed one row outside the rows with a stress and rho one row further out;
    // crop >= 3 keeps all of them inside the grid
    cudaError_t e;
    switch (D.storage) {
        case LBM_STORE_F16: e = launch_sweep<__half>(D, a, st); break;
        case LBM_STORE_BF16: e = launch_sweep<__nv_bfloat16>(D, a, st); break;
        default: e = launch_sweep<float>(D, a, st);
    }
    if (e != cudaSuccess) return e;
    reduce_kernel<<<kDiagTerms + (2 * (a.r1 - a.r0) + 7) / 8, 256, 0, st>>>(a, D.out);
    return cudaGetLastError();
}

cudaError_t launch_fields(const DiagLaunch& D, double* /*unused*/, cudaStream_t st) {
    (void)cudaGetLastError();
    DiagArgs a = make_args(D);
    cudaError_t e = moments(D, a, st);
    if (e != cudaSuccess) return e;
    dim3 grid((a.nx + DX - 1) / DX, (a.ny + BY - 1) / BY), block(DX, DY);
    velocity_kernel<<<grid, block, 0, st>>>(a);
    return cudaGetLastError();
}

}  // namespace lbm
