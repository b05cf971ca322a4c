// Collision of one site (Section 2 of arXiv 2101.04847: Eq. 1 moments,
// Shan-Chen + wall + buoyancy accelerations, forced BGK with the
// shifted-velocity equilibrium), shared by the step kernels.
//
// The two components are processed as the two lanes of float2 values with the
// packed FP32 instructions of this architecture (lattice.cuh): the collision is the
// same arithmetic for component A (lane x) and component B (lane y).
#pragma once
#include "lattice.cuh"

namespace lbm {

// Pseudopotentials of the eight neighbours, each as (B, A): lane x holds what acts on
// component A, lane y what acts on B.
struct Nbr2 { float2 E, W, N, S, NE, NW, SE, SW; };

// (sx, sy) = sum_i w_i psi'(x + c_i) c_i of the other component.
__device__ __forceinline__ void nbr_sum2(const Nbr2& p, float2& sx, float2& sy) {
    const float2 d = sub2(p.NE, p.SW);
    sx = fma2(splat(1.0f / 9.0f), sub2(p.E, p.W), mul2(splat(1.0f / 36.0f), add2(d, sub2(p.SE, p.NW))));
    sy = fma2(splat(1.0f / 9.0f), sub2(p.N, p.S), mul2(splat(1.0f / 36.0f), add2(d, sub2(p.NW, p.SE))));
}

// Common velocity u = sum_s j_s / tau_s / sum_s rho_s / tau_s (Eq. 1) and the
// accelerations a_s = F_s / rho_s: Shan-Chen coupling to the other component's
// pseudopotential, the external (buoyancy, body) accelerations and, on the wall
// rows, the fluid-boundary force.  False for a density below ph.rho_floor or a
// non-finite one: the caller raises bit 0 of the guard flag.  kWalls: the row may be a
// wall row.
template <bool kWalls>
__device__ __forceinline__ bool velocity_and_accel(float2 rho, float2 jx, float2 jy, const Nbr2& psi,
                                                   const Physics& ph, int y, int ny, float& ux, float& uy, float2& ax,
                                                   float2& ay) {
    const bool ok = rho.x >= ph.rho_floor[0] && rho.y >= ph.rho_floor[1] && rho.x < 1e30f && rho.y < 1e30f;
    // one product rounded, the other one not: spelled out, because the compiler may take either
    // and the results are not to depend on the kernel or the tile that a row falls into
    auto weighted = [&](float2 v) { return fmaf(v.x, ph.om[0], __fmul_rn(v.y, ph.om[1])); };
    const float inv = 1.0f / weighted(rho);
    ux = weighted(jx) * inv;
    uy = weighted(jy) * inv;
    float2 sx, sy;
    nbr_sum2(psi, sx, sy);
    ax = fma2(splat(-ph.G), sx, splat(ph.ax_ext));
    ay = fma2(splat(-ph.G), sy, make_float2(ph.ay_ext[0], ph.ay_ext[1]));
    if (kWalls && (y == 0 || y == ny - 1)) {
        if (y == 0) ay = add2(ay, make_float2(ph.ay_wall_bottom[0], ph.ay_wall_bottom[1]));
        if (y == ny - 1) ay = add2(ay, make_float2(ph.ay_wall_top[0], ph.ay_wall_top[1]));
        if (ph.wall_mirror) {
            // wall_mode 1: the virtual row beyond the wall holds this row's pseudopotentials
            // (the kernels passed zeros for it).  Its three neighbours add w c psi: the
            // straight one the other component's density here, the diagonals those at x + 1
            // and x - 1, i.e. (1/9) psi' + (1/36)(E' + W') along the outward normal and
            // (1/36)(E' - W') along x.
            const float2 own = swap2(rho);
            const float2 dn = fma2(splat(1.0f / 9.0f), own, mul2(splat(1.0f / 36.0f), add2(psi.E, psi.W)));
            const float2 dx = mul2(splat(1.0f / 36.0f), sub2(psi.E, psi.W));
            ax = fma2(splat(-ph.G), dx, ax);
            ay = fma2(splat(y == 0 ? ph.G : -ph.G), dn, ay);
        }
    }
    return ok;
}

// momenta (1 - 3) + (5 - 7) + (8 - 6) and (2 - 4) + (5 - 7) + (6 - 8)
__device__ __forceinline__ float2 momx2(const float2* f) {
    return add2(add2(sub2(f[1], f[3]), sub2(f[5], f[7])), sub2(f[8], f[6]));
}
__device__ __forceinline__ float2 momy2(const float2* f) {
    return add2(add2(sub2(f[2], f[4]), sub2(f[5], f[7])), sub2(f[6], f[8]));
}

// Equilibrium part shared by both collisions: feq_i = base_i + w_i rho u-terms,
// evaluated per pair of opposite directions (1,3), (2,4), (5,7), (6,8):
// f^eq_i + f^eq_ibar = 2 w (base + rho (9/2 (c.u')^2 - 3/2 u'^2)) and
// f^eq_i - f^eq_ibar = 6 w rho c.u'.  `k0` is the rest term, `sym(q, c)` the
// symmetric part of pair q.
template <typename Sym>
__device__ __forceinline__ void pairs2(float2 vx, float2 vy, float2 rho, Sym sym, float2 feq[9]) {
    const float2 c[4] = {vx, vy, add2(vx, vy), sub2(vy, vx)};
    const float w[4] = {1.0f / 9.0f, 1.0f / 9.0f, 1.0f / 36.0f, 1.0f / 36.0f};
    const int a[4] = {1, 2, 5, 6}, b[4] = {3, 4, 7, 8};
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const float2 s = sym(q, c[q]);
        const float2 anti = mul2(mul2(splat(w[q]), rho), mul2(splat(3.0f), c[q]));
        feq[a[q]] = add2(s, anti);
        feq[b[q]] = sub2(s, anti);
    }
}

// Forced BGK collision of one site (Section 2, Eqs. "Kinetic equation" and
// "Equilibrium distribution"): f <- f + (f^eq(rho_s, u + tau_s a_s) - f) / tau_s with
// a_s = F_s / rho_s computed directly (no division by rho_s).
//
// kExact (FP32 storage) works with the increments d_i = f*_i - f_i that the stored
// values really received (d_i is recomputed from the rounded f*_i; the subtraction
// is exact while |d_i| <= |f_i|, as in Dekker's Fast2Sum).  The BGK update changes a
// component's momentum by omega (rho_s u'_s - j_s) and its mass by nothing; the
// pairs 1/3 and 2/4 take half of the momentum defect each way, and the rest
// population takes minus the sum of the other eight increments.  The defects are
// sums of small increments, so their rounding is far below one unit in the last
// place of a population: mass is kept up to one rounding of f*_0 and the large,
// nearly cancelling inter-component Shan-Chen momenta do not random-walk the
// interface (plain FP32 moves rho by ~1e-5 of its range in 1000 steps at tau = 1).
// rho: the component densities, sum9_2(F).  Returns velocity_and_accel's verdict.
template <bool kExact, bool kWalls>
__device__ __forceinline__ bool collide_site(float2 F[9], float2 rho, const Nbr2& psi, const Physics& ph, int y, int ny) {
    const float2 jx = momx2(F), jy = momy2(F);
    float ux, uy;
    float2 ax, ay;
    const bool ok = velocity_and_accel<kWalls>(rho, jx, jy, psi, ph, y, ny, ux, uy, ax, ay);
    const float2 tau = make_float2(ph.tau[0], ph.tau[1]);
    const float2 om = make_float2(ph.om[0], ph.om[1]);
    const float2 vx = fma2(tau, ax, splat(ux));
    const float2 vy = fma2(tau, ay, splat(uy));
    // 1 - 3/2 u'^2
    const float2 omu = fma2(splat(-1.5f), fma2(vx, vx, mul2(vy, vy)), splat(1.0f));
    float2 feq[9];
    feq[0] = mul2(mul2(rho, splat(4.0f / 9.0f)), omu);
    const float2 r9 = mul2(rho, splat(1.0f / 9.0f)), r36 = mul2(rho, splat(1.0f / 36.0f));
    pairs2(vx, vy, rho,
           [&](int q, float2 c) { return mul2(q < 2 ? r9 : r36, fma2(mul2(splat(4.5f), c), c, omu)); }, feq);
    if (!kExact) {
#pragma unroll
        for (int i = 0; i < 9; ++i) F[i] = fma2(om, sub2(feq[i], F[i]), F[i]);
    } else {
        float2 in[5], d[9];
#pragma unroll
        for (int i = 1; i < 5; ++i) in[i] = F[i];
#pragma unroll
        for (int i = 1; i < 9; ++i) {
            const float2 o = fma2(om, sub2(feq[i], F[i]), F[i]);
            d[i] = sub2(o, F[i]);
            F[i] = o;
        }
        const float2 Jx = momx2(d), Jy = momy2(d);
        // (om (rho u' - j) - J) / 2, with om / 2 and -J / 2 exact scalings
        const float2 omh = mul2(om, splat(0.5f));
        const float2 hx = fma2(omh, fma2(rho, vx, mul2(jx, splat(-1.0f))), mul2(Jx, splat(-0.5f)));
        const float2 hy = fma2(omh, fma2(rho, vy, mul2(jy, splat(-1.0f))), mul2(Jy, splat(-0.5f)));
        F[1] = add2(F[1], hx);
        F[3] = sub2(F[3], hx);
        F[2] = add2(F[2], hy);
        F[4] = sub2(F[4], hy);
#pragma unroll
        for (int i = 1; i < 5; ++i) d[i] = sub2(F[i], in[i]);
        const float2 m = add2(add2(add2(d[1], d[2]), add2(d[3], d[4])), add2(add2(d[5], d[6]), add2(d[7], d[8])));
        F[0] = sub2(F[0], m);
    }
    return ok;
}

// The same collision on shifted populations h_i = f_i - w_i rho0_s (16-bit
// storage), without forming f: rho_s = rho0_s + sum_i h_i, j_s = sum_i c_i h_i
// (the shift carries no momentum), and
//   f^eq_i - w_i rho0_s = w_i (rho_s - rho0_s) + w_i rho_s (9/2 (c_i.u')^2 - 3/2 u'^2 + 3 c_i.u'),
// so h_i <- h_i + (f^eq_i - w_i rho0_s - h_i) / tau_s.
// dr = sum9_2(H).
template <bool kWalls>
__device__ __forceinline__ bool collide_shifted(float2 H[9], float2 dr, const Nbr2& psi, const Physics& ph, int y,
                                                int ny) {
    const float2 rho = add2(make_float2(ph.shift[0], ph.shift[1]), dr);
    const float2 jx = momx2(H), jy = momy2(H);
    float ux, uy;
    float2 ax, ay;
    const bool ok = velocity_and_accel<kWalls>(rho, jx, jy, psi, ph, y, ny, ux, uy, ax, ay);
    const float2 tau = make_float2(ph.tau[0], ph.tau[1]);
    const float2 om = make_float2(ph.om[0], ph.om[1]);
    const float2 vx = fma2(tau, ax, splat(ux));
    const float2 vy = fma2(tau, ay, splat(uy));
    const float2 usq = mul2(splat(1.5f), fma2(vx, vx, mul2(vy, vy)));
    const float2 mrho = mul2(rho, splat(-1.0f));
    float2 feq[9];
    feq[0] = mul2(splat(4.0f / 9.0f), fma2(mrho, usq, dr));
    pairs2(vx, vy, rho,
           [&](int q, float2 c) {
               const float w = q < 2 ? 1.0f / 9.0f : 1.0f / 36.0f;
               return mul2(splat(w), fma2(rho, fma2(mul2(splat(4.5f), c), c, mul2(usq, splat(-1.0f))), dr));
           },
           feq);
#pragma unroll
    for (int i = 0; i < 9; ++i) H[i] = fma2(om, sub2(feq[i], H[i]), H[i]);
    return ok;
}

}  // namespace lbm
