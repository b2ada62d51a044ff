// lbm_kernels.cuh -- kernels of one time step (template definitions; each
// storage type is instantiated in its own translation unit).
//
//   k_collide_d2q9   the whole time step in one persistent launch: every
//                    warp walks row tiles of 32 x VEC sites (pull-stream +
//                    moments + f* + dS + LBGK), the block keeps the k best
//                    of its sites with dS > delta, and the block that
//                    finishes last selects the k largest dS of all blocks'
//                    and makes the Ehrenfests' step f <- f* at those sites
//                    (Sec. 3.2; (ESLB)).  No block waits for another.
//   k_collide_d2q9_tma   the same step with the sources of block tiles
//                    staged in shared memory by bulk tensor copies
//   k_collide_site   the same step, one site per thread (D1Q3)
//   k_tube           many steps of a short D1Q3 run in one launch (one cluster)
//   k_select         the selection as a stand-alone kernel (test hook)
#pragma once

#include <algorithm>

#include <cooperative_groups.h>
#include <cuda.h>

#include "lbm_device.cuh"
#include "lbm_rendezvous.h"
#include "lbm_energy.cuh"
#include "lbm_mlp.cuh"
#include "lbm_internal.h"

namespace lbm {

constexpr int kSelectThreads = 1024;
constexpr int kSiteBlock = 64;       // one site per thread: FP64 work over as many SMs as there are blocks
constexpr int kStage = 1024;         // candidates staged in shared memory by the last block

template <typename L, typename T, int EQ>
__device__ __forceinline__ void equilibrium(const Params& P, T drho, T rho, T ux, T uy, T* gs) {
    (void)P;
    if constexpr (EQ == EQ_POLY) feq_poly<L, T>(drho, rho, ux, uy, gs);
    else feq_entropic<L, T, kF64<T>>(drho, rho, ux, uy, gs);   // (FP64 storage: rho0 = 0)
}

// Energy-constrained entropic f* (D2Q9 only) as deviations from the
// moments (drho, j, 2E); Newton from the energy multiplier's start mu3 (the
// network's warm start in the learned form, else 0: the polynomial start
// point (3 u_x, 3 u_y, 0), the multipliers of the first-order expansion about
// rest; the momentum multipliers follow in closed form).
template <typename T, int EQ>
__device__ __forceinline__ void equilibrium_energy(T rho, T jx, T jy, T e2, T* gs, NewtonCount& nc,
                                                   float mu3 = 0.0f) {
    if constexpr (sizeof(T) == 4) {
        // FP32 / FP16 storage: the float-float finish (no FP64 work)
        energy_solve_ff(rho, jx, jy, e2, mu3, gs, nc);
    } else {
        // FP64 storage (rho0 = 0): FP64 finish to 4e-15 (the FP64 parity bound)
        const double ir = recip<double>(rho);
        energy_solve(rho, jx * ir, jy * ir, e2 * ir, mu3, gs, nc, 4e-15f);
    }
}

template <typename L, typename T>
__device__ __forceinline__ void moments(const T* g, T rho0, T& drho, T& rho, T& jx, T& jy) {
    if constexpr (L::Q == 9 && kF64<T>) {
        // sums of the diagonals shared (16 additions)
        const T pe = g[5] + g[8], pw = g[6] + g[7];
        jx = (g[1] - g[3]) + (pe - pw);
        jy = (g[2] - g[4]) + ((g[5] - g[8]) + (g[6] - g[7]));
        drho = g[0] + ((g[1] + g[3]) + (g[2] + g[4])) + (pe + pw);
    } else if constexpr (L::Q == 9) {
        // pairwise sums (D2Q9 numbering: 1..4 E N W S, 5..8 NE NW SW SE)
        drho = ((g[0] + g[1]) + (g[2] + g[3])) + ((g[4] + g[5]) + (g[6] + g[7])) + g[8];
        jx = ((g[1] - g[3]) + (g[5] - g[6])) + (g[8] - g[7]);
        jy = ((g[2] - g[4]) + (g[5] - g[8])) + (g[6] - g[7]);
    } else {
        // D1Q3: 0 rest, 1 left, 2 right
        drho = (g[0] + g[1]) + g[2];
        jx = g[2] - g[1];
        jy = T(0);
    }
    rho = rho0 + drho;
}

// u = j / rho by the refined reciprocal (recip).
template <typename T>
__device__ __forceinline__ void velocity(T jx, T jy, T rho, T& ux, T& uy) {
    const T r = recip<T>(rho);
    ux = jx * r;
    uy = jy * r;
}

// Whether rho, u_x and u_y are finite.
__device__ __forceinline__ bool all_finite(float rho, float ux, float uy) { return isfinite(rho + ux + uy); }
__device__ __forceinline__ bool all_finite(double rho, double ux, double uy) {
    // exponent fields (integer operations)
    const int a = __double2hiint(rho), b = __double2hiint(ux), c = __double2hiint(uy);
    return ((a & 0x7ff00000) != 0x7ff00000) & ((b & 0x7ff00000) != 0x7ff00000) & ((c & 0x7ff00000) != 0x7ff00000);
}

// Polynomial D2Q9 f* of FP64 storage (rho0 = 0) from the moments: with
// j = rho u the terms of feq_poly need neither rho nor products of it (30
// FP64 operations instead of 37).
__device__ __forceinline__ void feq_poly_f64(double rho, double jx, double jy, double ux, double uy, double* gs) {
    const double c0 = fma(-1.5, fma(jx, ux, jy * uy), rho);
    const double ca = c0 * (1.0 / 9.0), cb = c0 * (1.0 / 36.0);
    gs[0] = c0 * (4.0 / 9.0);
    double a = fma(0.5 * jx, ux, ca), b = jx * (1.0 / 3.0);
    gs[1] = a + b;
    gs[3] = a - b;
    a = fma(0.5 * jy, uy, ca);
    b = jy * (1.0 / 3.0);
    gs[2] = a + b;
    gs[4] = a - b;
    double j = jx + jy;
    a = fma(0.125 * j, ux + uy, cb);
    b = j * (1.0 / 12.0);
    gs[5] = a + b;
    gs[7] = a - b;
    j = jx - jy;
    a = fma(0.125 * j, ux - uy, cb);
    b = j * (1.0 / 12.0);
    gs[8] = a + b;
    gs[6] = a - b;
}

// 2E = sum |v|^2 f = sum |v|^2 g + rho0 sum W |v|^2 of a site's deviations.
template <typename L, typename T>
__device__ __forceinline__ T energy_moment(const T* g, T rho0) {
    T e2 = T(L::sum_w_c2) * rho0;
#pragma unroll
    for (int i = 0; i < L::Q; i++)
        if (L::cx(i) * L::cx(i) + L::cy(i) * L::cy(i) == 1) e2 = e2 + g[i];
        else if (L::cx(i) * L::cx(i) + L::cy(i) * L::cy(i) == 2) e2 = e2 + T(2) * g[i];
    return e2;
}

// Quasiequilibrium of a gathered site (shared by the collision, the
// Ehrenfests' step and the exports so that all round identically).  mu3:
// start of the energy forms' multiplier (0: the polynomial start).
template <typename L, typename T, int EQ>
__device__ __forceinline__ void site_equilibrium(const Params& P, const T* g, T* gs, T& rho, T& ux,
                                                 T& uy, NewtonCount& nc, float mu3 = 0.0f) {
    T drho, jx, jy;
    moments<L, T>(g, Par<T>::rho0(P), drho, rho, jx, jy);
    if constexpr (kF64<T>) rho = drho;   // FP64 storage holds f itself (rho0 = 0)
    velocity<T>(jx, jy, rho, ux, uy);
    if constexpr (EQ == EQ_POLY && L::Q == 9 && kF64<T>) {
        (void)nc;
        (void)mu3;
        feq_poly_f64(rho, jx, jy, ux, uy, gs);
    } else if constexpr (EQ >= EQ_ENERGY) {
        const T e2 = energy_moment<L, T>(g, Par<T>::rho0(P));
        equilibrium_energy<T, EQ>(rho, jx, jy, e2, gs, nc, mu3);
    } else {
        (void)nc;
        (void)mu3;
        equilibrium<L, T, EQ>(P, drho, rho, ux, uy, gs);
    }
}
template <typename L, typename T, int EQ>
__device__ __forceinline__ void site_equilibrium(const Params& P, const T* g, T* gs, T& rho, T& ux,
                                                 T& uy) {
    NewtonCount nc = {0, 0, 0, 0};
    site_equilibrium<L, T, EQ>(P, g, gs, rho, ux, uy, nc);
}

// Per-thread Newton counts flushed to the run's statistics (energy forms).
__device__ __forceinline__ void flush_newton(const Params& P, NewtonCount& nc) {
    unsigned v[4] = {nc.it32, nc.it64, nc.sites, nc.fails};
#pragma unroll
    for (int j = 0; j < 4; j++) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v[j] += __shfl_xor_sync(0xffffffffu, v[j], o);
    }
    if ((threadIdx.x & 31) == 0 && v[2] > 0) {
        for (int j = 0; j < 4; j++) atomicAdd(P.newton_stats + j, (unsigned long long)v[j]);
        if (v[3] > 0) atomicOr(P.err, ERR_NEWTON);
    }
}

// FP64 recomputation of dS from the stored populations (precision form).
template <typename L, typename T, int EQ>
__device__ __noinline__ double delta_s_fp64(PopArr<L::Q, T> g, double rho0) {
    double gd[L::Q], gs[L::Q], drho, rho, jx, jy, ux, uy;
#pragma unroll
    for (int i = 0; i < L::Q; i++) gd[i] = (double)g.v[i];
    moments<L, double>(gd, rho0, drho, rho, jx, jy);
    velocity<double>(jx, jy, rho, ux, uy);
    if constexpr (EQ >= EQ_ENERGY) {
        double e2 = L::sum_w_c2 * rho0;
#pragma unroll
        for (int i = 0; i < L::Q; i++) e2 += (double)(L::cx(i) * L::cx(i) + L::cy(i) * L::cy(i)) * gd[i];
        double fs[9];
        NewtonCount nc = {0, 0, 0, 0};
        energy_solve(rho, ux, uy, e2 / rho, 0.0f, fs, nc, 4e-15f);
#pragma unroll
        for (int i = 0; i < L::Q; i++) gs[i] = fs[i] - L::w(i) * rho0;
    } else if constexpr (EQ == EQ_POLY) {
        feq_poly<L, double>(drho, rho, ux, uy, gs);
    } else {
        feq_entropic<L, double>(drho, rho, ux, uy, gs);
    }
    return delta_s_exact<L, double>(gd, gs, rho0);
}

// Per-site update after the gather: moments, f*, the dS bound, LBGK.
// g: pre-collision deviations in, post-collision deviations out.
// Returns true when the bound does not clear the site (dS may exceed delta):
// its exact dS is then evaluated later from the unchanged source field.
// ELBM (elbmLB): alpha with S(f + alpha (f* - f)) = S(f) for one site, from
// the full populations f and f*, in the arithmetic U of the storage (FP64
// to 1e-15 relative for FP64 storage; FP32 to its rounding for FP32 and
// FP16 storage, whose populations carry FP32 rounding already).  With
// D = f* - f and x_i = D_i / f_i the condition is
// G(a) = sum f_i phi(a x_i) - a R = 0, R = sum D_i log1p(x_i) (sum D = 0 and
// ln f* linear in the conserved moments remove the two entropies'
// cancellation); G is convex, G(0) = 0, G(1) <= 0, so the root in
// [1, alpha_max] (alpha_max = 1 / max(-x_i): f + a D >= 0) is unique.
// Newton with G'(a) = sum D_i log1p(a x_i) - R, falling back to bisection
// whenever a step leaves the bracket.  The start point is the root of the
// series of G to second order in x, a = 2 + S3 / (3 S2) with
// Sn = sum f_i x_i^n; near equilibrium (max |x| < 0.1, so alpha_max > 10)
// the bracket check at alpha_max is skipped.  Stop: FP64 when a step or the
// bracket falls below 1e-15 relative; FP32 once a step is below 3e-4
// relative (Newton converges quadratically with G''/G' ~ 1/2 here, so the
// result of that step is within about 1e-7 of the root, FP32's rounding;
// iterating further in FP32 only chases the rounding noise of G, and the
// slowest lane holds its whole warp).  a = 2 when f = f*; alpha_max when
// the entropy still exceeds S(f) there; -1 when some f_i or f*_i is not
// positive.
// Near equilibrium (max |x| < 0.1, almost every site) both precisions take
// a branch-free path instead: with Sn = sum f_i x_i^n, the series of G / a is
//   P(a) = sum_{n>=2} (-1)^n Sn (a^{n-1}/n - 1)/(n - 1),
// whose terms beyond n = 10 are below 1e-9 S2 for |a x| <= 0.21 (the root
// lies within 2 +- max|x| / 3 there), far below FP32's rounding of P (about
// 1e-7 S2), and beyond n = 24 below 1e-18 S2, under FP64's; Newton steps on
// P from the series root 2 + S3 / (3 S2) (three in FP32, four in FP64: P is
// almost linear, P' ~ S2 / 2, and the start is off by O(max|x|^2)) reach the
// root.  No logarithm and no data-dependent loop, so the lanes of a warp stay
// together.  For max |x| < 1/64 (whole warps of it away from the cylinder and
// its wake) shorter sums reach the same rounding: with |a x| <= 0.033 the terms
// beyond n = 6 are below 2e-9 S2 (FP32), beyond n = 13 below 1e-18 S2 (FP64),
// and the start is off by 2e-4 at most, so two steps (FP64: three) do.  2048 x
// 1024, FP32: 85 -> 51 us per step.
template <int Q, int NT, int ITERS, typename U>
__device__ __forceinline__ U elbm_alpha_series(const U* D, const U* x) {
    // c_n = (-1)^n Sn / (n - 1), n = 2..NT, with Sn = sum D_i x_i^{n-1}
    U c[NT + 1];
#pragma unroll
    for (int n = 0; n <= NT; n++) c[n] = U(0);
#pragma unroll
    for (int i = 0; i < Q; i++) {
        U t = D[i] * x[i];
#pragma unroll
        for (int n = 2; n <= NT; n++) {
            c[n] += t;
            t *= x[i];
        }
    }
    if (!(c[2] > U(sizeof(U) == 8 ? 1e-290 : 1e-30))) return U(2);   // (below: f = f* to rounding)
    const U a0 = U(2) + c[3] * recip<U>(U(3) * c[2]);   // 2 + S3 / (3 S2)
    // P(a) = a B(a) - sum c_n with B(a) = sum b_n a^{n-2}, b_n = c_n / n;
    // P'(a) = sum d_n a^{n-2}, d_n = c_n (n - 1) / n
    U b[NT + 1], d[NT + 1], sumc = U(0);
#pragma unroll
    for (int n = 2; n <= NT; n++) {
        const U cn = ((n & 1) ? -c[n] : c[n]) * U(1.0 / (n - 1));
        sumc += cn;
        b[n] = cn * U(1.0 / n);
        d[n] = cn * U((n - 1.0) / n);
    }
    U a = a0;
#pragma unroll
    for (int it = 0; it < ITERS; it++) {
        U B = b[NT], dP = d[NT];
#pragma unroll
        for (int n = NT - 1; n >= 2; n--) {
            B = dfma<U>(B, a, b[n]);
            dP = dfma<U>(dP, a, d[n]);
        }
        a -= (a * B - sumc) * recip<U>(dP);
    }
    return a;
}

template <typename L, typename U>
__device__ __noinline__ U elbm_alpha(const U* f, const U* fs) {
    constexpr bool fp64 = sizeof(U) == 8;
    constexpr U step_tol = fp64 ? U(1e-15) : U(3e-4);
    constexpr U bracket_tol = fp64 ? U(1e-15) : U(4.0 * 1.1920929e-7);
    constexpr int max_it = fp64 ? 100 : 40;
    U D[L::Q], x[L::Q], R = U(0), xneg = U(0), s2 = U(0), s3 = U(0), xm = U(0);
    bool moved = false, positive = true;
#pragma unroll
    for (int i = 0; i < L::Q; i++) {
        positive &= f[i] > U(0) && fs[i] > U(0);
        D[i] = fs[i] - f[i];
        moved |= D[i] != U(0);
        x[i] = D[i] * recip<U>(f[i]);
        xneg = fmax(xneg, -x[i]);
        xm = fmax(xm, fabs(x[i]));
    }
    if (!positive) return U(-1);
    if (!moved || !(xneg > U(0))) return U(2);
    // near equilibrium the series path: terms to n = 10 reach FP32's rounding,
    // to n = 24 FP64's (the omitted terms are below 1e-18 S2 for |a x| <= 0.21)
    if (xm < U(1.0 / 64.0)) return elbm_alpha_series<L::Q, fp64 ? 13 : 6, fp64 ? 3 : 2, U>(D, x);
    if (xm < U(0.1)) return elbm_alpha_series<L::Q, fp64 ? 24 : 10, fp64 ? 4 : 3, U>(D, x);
#pragma unroll
    for (int i = 0; i < L::Q; i++) {
        R += D[i] * log1p(x[i]);
        s2 += D[i] * x[i];
        s3 += D[i] * x[i] * x[i];
    }
    if (!(R > U(0))) return U(2);
    const U amax = U(1) / xneg;
    auto G = [&](U a) {
        U s = U(0);
#pragma unroll
        for (int i = 0; i < L::Q; i++) s += f[i] * phi_fn<U>(a * x[i]);
        return s - a * R;
    };
    U lo = U(1), hi = amax;
    if (!(xm < U(0.1)) && G(hi) <= U(0)) return hi;
    U a = U(2) + s3 / (U(3) * s2);
    if (!(a > lo && a < hi)) a = U(0.5) * (lo + hi);
    for (int it = 0; it < max_it; it++) {
        const U g = G(a);
        if (g <= U(0)) lo = a;
        else hi = a;
        U dg = -R;
#pragma unroll
        for (int i = 0; i < L::Q; i++) dg += D[i] * log1p(a * x[i]);
        U na = a - g / dg;
        const bool newton = na > lo && na < hi;
        if (!newton) na = U(0.5) * (lo + hi);
        const bool done = (newton && fabs(na - a) <= step_tol * a) || hi - lo <= bracket_tol * hi;
        a = na;
        if (done) break;
    }
    return a;
}

// The ELBM step factor -alpha beta of a site from its deviations (kept out
// of line: the LBGK path does not carry its arrays).
template <typename L, typename T>
__device__ __noinline__ T elbm_factor(PopArr<L::Q, T> g, PopArr<L::Q, T> gs, T rho0, T beta) {
    T fd[L::Q], fsd[L::Q];
#pragma unroll
    for (int i = 0; i < L::Q; i++) {
        fd[i] = g.v[i] + T(L::w(i)) * rho0;
        fsd[i] = gs.v[i] + T(L::w(i)) * rho0;
    }
    T a = elbm_alpha<L, T>(fd, fsd);
    if (a < T(0)) a = T(2);   // outside the positive cone: dS = +inf, LBGK
    return -a * beta;
}

// Exact dS of a site from its pre-collision deviations g and its
// quasiequilibrium gs (rho0, dl: the run's rho0 and delta in T).  The
// precision form (recheck) decides the sites whose FP32 dS lies within band
// of delta (a bound on the FP32 evaluation error of dS, set by the host) in
// FP64; the value kept for ranking then stays on the same side of delta.
// Returns dS in T (NaN for a non-finite state).  Out of line: the sites the
// bound does not clear are few, and the update path keeps its registers.
template <typename L, typename T, int EQ>
__device__ __forceinline__ T recheck_ds(const PopArr<L::Q, T>& g, T ds, T dl, double delta, double rho0d, double band,
                                        int recheck) {
    if (recheck && isfinite(ds) && fabs((double)ds - delta) <= band) {
        const double d64 = delta_s_fp64<L, T, EQ>(g, rho0d);
        if (d64 > delta) ds = (T)d64 > dl ? (T)d64 : nextafter(dl, T(INFINITY));
        else ds = T(-1);
    }
    return ds;
}
template <typename L, typename T, int EQ>
__device__ __noinline__ T resolved_ds(PopArr<L::Q, T> g, PopArr<L::Q, T> gs, T rho0, T dl, double delta,
                                      double rho0d, double band, int recheck) {
    return recheck_ds<L, T, EQ>(g, delta_s_exact<L, T>(g.v, gs.v, rho0), dl, delta, rho0d, band, recheck);
}

// The same from the site's pre-collision deviations g and quasiequilibrium
// gs already at hand.
template <typename L, typename T, int EQ>
__device__ __forceinline__ T site_ds(const Params& P, const T* g, const T* gs) {
    PopArr<L::Q, T> ga, gsa;
#pragma unroll
    for (int i = 0; i < L::Q; i++) {
        ga.v[i] = g[i];
        gsa.v[i] = gs[i];
    }
    return resolved_ds<L, T, EQ>(ga, gsa, Par<T>::rho0(P), Par<T>::delta(P), P.delta, P.rho0, P.recheck_band,
                                 P.recheck);
}

// A ghost column of a slab (a copy of a neighbour's sites: never a candidate).
__device__ __forceinline__ bool ghost_column(const Params& P, int x) {
    return P.slab && (x < P.own_x0 || x >= P.own_x1);
}

// PROBE = false: the caller guarantees the site is not the probe site.
// PROJ: remove the rounding defects of the conserved moments of f - f*
// (conserve_neq; FP32 storage).  g leaves as the deviations to store, before
// the storage's rounding (store_round).  RESOLVE: a site the bound does not
// clear has its dS evaluated here, from the pre-collision g and f* at hand
// (site_ds), and stored to *ds_out (-1 for every other site, and for a
// slab's ghost columns).  gs_out (optional): f*, for a caller that resolves
// the site itself.
template <typename L, typename T, int EQ, bool PROJ, bool PROBE = true, bool RESOLVE = false>
__device__ __forceinline__ bool update_site(const Params& P, T* g, int x, int y, long long t,
                                            bool& nonfinite, NewtonCount& nc,
                                            float mu3 = 0.0f, T* ds_out = nullptr, T* gs_out = nullptr) {
    T gs[L::Q], rho, ux, uy;
    site_equilibrium<L, T, EQ>(P, g, gs, rho, ux, uy, nc, mu3);
    nonfinite |= !all_finite(rho, ux, uy);
    if (PROBE && x == P.probe_x && y == P.probe_y && P.probe_ring)
        P.probe_ring[t % P.ring_cap] = (double)ux;
    if (gs_out) {
#pragma unroll
        for (int i = 0; i < L::Q; i++) gs_out[i] = gs[i];
    }
    T d[L::Q];
#pragma unroll
    for (int i = 0; i < L::Q; i++) d[i] = g[i] - gs[i];
    if constexpr (PROJ) conserve_neq<L, EQ>(d);
    // (no short-circuit: the site's update stays one branch-free block)
    const bool pending =
        (P.k > 0) & !ds_cleared<L, T, EQ>(d, gs, rho, ux, uy, Par<T>::rho0(P), Par<T>::delta(P));
    if constexpr (RESOLVE) {
        T ds = T(-1);
        if (pending && !ghost_column(P, x)) ds = site_ds<L, T, EQ>(P, g, gs);
        *ds_out = ds;
    }
    T nb2 = T(-2) * Par<T>::beta(P);
    if constexpr (EQ == EQ_ENTROPIC) {
        if (P.elbm) {
            // f' = f + alpha beta (f* - f) (elbmLB)
            PopArr<L::Q, T> ga, gsa;
#pragma unroll
            for (int i = 0; i < L::Q; i++) {
                ga.v[i] = g[i];
                gsa.v[i] = gs[i];
            }
            nb2 = elbm_factor<L, T>(ga, gsa, Par<T>::rho0(P), Par<T>::beta(P));
        }
    }
#pragma unroll
    for (int i = 0; i < L::Q; i++) g[i] = dfma<T>(nb2, d[i], g[i]);
    return pending;
}

// update_site of two adjacent sites at once in packed FP32 arithmetic (FP32
// and FP16 storage; every operation the scalar one's, half by half).  nc, mu3:
// the sites' Newton counts and start points (energy forms).  g: pre-collision deviations in,
// post-collision deviations out, before the storage's rounding.  Returns bit 0
// / bit 1: the bound does not clear the first / second site.
// The scalar update issues about 240 instructions per site, 145 of them FP32
// arithmetic, which packed take half the slots.  64 steps of 4096 x 2048 and
// the export: FP16 4911 -> 4602 us, polynomial FP32 (bound by memory) 6314 ->
// 6165 us; 1531 x 765 entropic FP32 1208 -> 1143 us.
template <typename S, int EQ>
__device__ __forceinline__ unsigned update_pair(const Params& P, f2* g, bool& nonfinite, NewtonCount* nc = nullptr,
                                                f2 mu3 = f2(0.0f)) {
    using L = D2Q9;
    static_assert(sizeof(typename Store<S>::T) == 4, "FP32 arithmetic");
    f2 gs[L::Q], drho, rho, jx, jy, ux, uy;
    moments<L, f2>(g, f2(P.rho0f), drho, rho, jx, jy);
    velocity<f2>(jx, jy, rho, ux, uy);
    if constexpr (EQ >= EQ_ENERGY) energy_solve_pair(rho, jx, jy, energy_moment<L, f2>(g, f2(P.rho0f)), mu3, gs, nc);
    else equilibrium<L, f2, EQ>(P, drho, rho, ux, uy, gs);
    const f2 s = (rho + ux) + uy;
    nonfinite |= !isfinite(s.x) | !isfinite(s.y);
    f2 d[L::Q];
#pragma unroll
    for (int i = 0; i < L::Q; i++) d[i] = g[i] - gs[i];
    if constexpr (Store<S>::kProject) conserve_neq<L, EQ>(d);
    const unsigned pending =
        P.k > 0 ? 3u & ~ds_cleared_pair<L, EQ>(d, gs, rho, ux, uy, P.rho0f, P.deltaf) : 0u;
    f2 nb2(-2.0f * P.betaf);
    if constexpr (EQ == EQ_ENTROPIC) {
        if (P.elbm) {
            PopArr<L::Q, float> a, b, as, bs;
#pragma unroll
            for (int i = 0; i < L::Q; i++) {
                a.v[i] = g[i].x;
                b.v[i] = g[i].y;
                as.v[i] = gs[i].x;
                bs.v[i] = gs[i].y;
            }
            nb2.x = elbm_factor<L, float>(a, as, P.rho0f, P.betaf);
            nb2.y = elbm_factor<L, float>(b, bs, P.rho0f, P.betaf);
        }
    }
#pragma unroll
    for (int i = 0; i < L::Q; i++) g[i] = f2_fma(nb2, d[i], g[i]);
    return pending;
}

// Shared copy of the network in the learned form's kernels (empty otherwise).
template <int EQ> struct MlpSlot {
    __device__ void fill(const Params&) {}
};
template <> struct MlpSlot<EQ_ENERGY_MLP> {
    MlpSmemQ s;
    __device__ void fill(const Params& P) {
        mlp_fill(s, P.mlp);
        mlp_fill_quads(s, P.mlp);
    }
};

// Learned form: the network's start of the energy multiplier for the warp's
// 32 sites (lane l: its gathered site g, or valid = false).  Every lane must
// call it.
template <typename T>
__device__ __forceinline__ float mlp_site_start(const Params& P, const MlpSmemQ& ms, bool valid, const T* g) {
    float rho = 1.0f, ux = 0.0f, uy = 0.0f, e2 = 0.0f;
    if (valid) {
        T drho, r, jx, jy;
        moments<D2Q9, T>(g, Par<T>::rho0(P), drho, r, jx, jy);
        rho = (float)r;
        const float ir = 1.0f / rho;
        ux = (float)jx * ir;
        uy = (float)jy * ir;
        e2 = (float)energy_moment<D2Q9, T>(g, Par<T>::rho0(P));
        valid = rho > 0.0f && isfinite(rho + ux + uy + e2);
    }
    return mlp_start(ms, rho, ux, uy, e2, valid);
}

// Exact dS of site (x, y) with the pre-collision state re-gathered from the
// source field (not written during a step); -1 on a slab's ghost column.
template <typename L, typename S, int EQ>
__device__ __noinline__ typename Store<S>::T resolve_ds(const Params& P, int x, int y) {
    using T = typename Store<S>::T;
    if (ghost_column(P, x)) return T(-1);
    T g[L::Q], gs[L::Q], rho, ux, uy;
    gather_site<L, S>(P, x, y, g);
    site_equilibrium<L, T, EQ>(P, g, gs, rho, ux, uy);
    return site_ds<L, T, EQ>(P, g, gs);
}

// Warp-level append of candidates (sites with dS > delta) to the global
// list: one ballot, one atomic per warp when any lane has a candidate.
// Every lane of the warp must call it.
template <typename T>
__device__ __forceinline__ void warp_push(const Params& P, bool cand, T ds, unsigned site) {
    const unsigned m = __ballot_sync(0xffffffffu, cand);
    if (m == 0) return;
    const int lane = threadIdx.x & 31;
    unsigned base = 0;
    if (lane == 0) base = atomicAdd(P.cand_count, (unsigned)__popc(m));
    base = __shfl_sync(0xffffffffu, base, 0);
    if (cand) {
        const unsigned slot = base + __popc(m & ((1u << lane) - 1u));
        P.cand_key[slot] = ds_key((double)ds);
        P.cand_idx[slot] = site;
    }
}

// ---------------------------------------------------------------------------
// Block stage of the selection (k sites of the whole grid are selected, so a
// block never contributes more than its own k best): a block holds its
// candidates in shared memory, cuts them to its k largest (dS, -index) with
// the block radix select whenever the buffer fills, and flushes what it kept
// to the global list when it ends.  The global select then ranks at most
// k x blocks keys.  With k too large for a cut to free room, the block
// flushes its buffer to the global list instead (which holds one slot per
// site and cannot overflow).  CAP entries: room for the entries kept by a
// cut plus one round of appends (a round of pending sites resolved by the
// block, or the sites of one staged tile).
// ---------------------------------------------------------------------------
constexpr int kBlockCand = 320;   // room for a round of 256 candidates above a cut

template <int CAP>
struct BlockCandT {
    static constexpr int kCap = CAP;
    unsigned long long key[CAP];
    unsigned idx[CAP];
    unsigned n;          // candidates appended (entries beyond CAP went to the global list)
    unsigned base;
};
using BlockCand = BlockCandT<kBlockCand>;

// Warp-level append to the block's buffer (every lane calls).  Returns the
// number of candidates the warp appended (the same on every lane).
template <typename T, int CAP>
__device__ __forceinline__ unsigned block_push(const Params& P, BlockCandT<CAP>& bc, bool cand, T ds,
                                               unsigned site) {
    const unsigned m = __ballot_sync(0xffffffffu, cand);
    if (m == 0) return 0u;
    const int lane = threadIdx.x & 31;
    unsigned base = 0;
    if (lane == 0) base = atomicAdd(&bc.n, (unsigned)__popc(m));
    base = __shfl_sync(0xffffffffu, base, 0);
    if (cand) {
        const unsigned slot = base + __popc(m & ((1u << lane) - 1u));
        const unsigned long long key = ds_key((double)ds);
        if (slot < (unsigned)CAP) {
            bc.key[slot] = key;
            bc.idx[slot] = site;
        } else {
            // no room (the global list has room for every site)
            const unsigned g = atomicAdd(P.cand_count, 1u);
            P.cand_key[g] = key;
            P.cand_idx[g] = site;
        }
    }
    return (unsigned)__popc(m);
}

// Keep the k best of the buffer (all threads call; blockDim >= 128, or at most
// kPer entries per thread).  This and block_flush below return past a barrier
// that follows every thread's read of the count, so that a caller may go on to
// append at once: otherwise a warp that returned early could raise the count
// before a slower one has read it, and the two would take different branches,
// and barriers, from there on.
template <int CAP>
__device__ __noinline__ void block_cut(BlockCandT<CAP>& bc, TopkScratch& sc, int k) {
    constexpr int kPer = (CAP + 127) / 128;
    const int tid = threadIdx.x, nt = blockDim.x;
    __syncthreads();
    const int n = (int)min(bc.n, (unsigned)CAP);
    if (n <= k) {   // uniform: n was read after the barrier
        __syncthreads();
        return;
    }
    const Thresh th = block_topk(sc, n, k, [&](int e) { return bc.key[e]; }, [&](int e) { return bc.idx[e]; });
    unsigned long long kk[kPer];
    unsigned ii[kPer];
    bool keep[kPer];
#pragma unroll
    for (int r = 0; r < kPer; r++) {
        const int e = tid + r * nt;
        keep[r] = e < n && th.selected(bc.key[e], bc.idx[e]);
        kk[r] = keep[r] ? bc.key[e] : 0ull;
        ii[r] = keep[r] ? bc.idx[e] : 0u;
    }
    __syncthreads();
    if (tid == 0) bc.n = 0;
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kPer; r++) {
        if (keep[r]) {
            const unsigned slot = atomicAdd(&bc.n, 1u);
            bc.key[slot] = kk[r];
            bc.idx[slot] = ii[r];
        }
    }
    __syncthreads();
}

// Move the buffer to the global candidate list (all threads call).
template <int CAP>
__device__ __noinline__ void block_flush(const Params& P, BlockCandT<CAP>& bc) {
    __syncthreads();
    const int n = (int)min(bc.n, (unsigned)CAP);
    if (n == 0) {   // uniform
        __syncthreads();
        return;
    }
    if (threadIdx.x == 0) bc.base = atomicAdd(P.cand_count, (unsigned)n);
    __syncthreads();
    const unsigned base = bc.base;
    for (int e = threadIdx.x; e < n; e += blockDim.x) {
        P.cand_key[base + e] = bc.key[e];
        P.cand_idx[base + e] = bc.idx[e];
    }
    __syncthreads();
    if (threadIdx.x == 0) bc.n = 0;
    __syncthreads();
}

// Make room for another blockDim candidates (all threads call).
template <int CAP>
__device__ __forceinline__ void block_room(const Params& P, BlockCandT<CAP>& bc, TopkScratch& sc) {
    const int room = CAP - (int)blockDim.x;
    __syncthreads();
    const bool full = (int)bc.n > room;
    __syncthreads();   // every thread has read the count before any appends
    if (full) {   // uniform
        if (P.k <= room) block_cut(bc, sc, P.k);
        else block_flush(P, bc);
    }
}

// What the block contributes to the global select: its k best (all threads).
template <int CAP>
__device__ __forceinline__ void block_finish(const Params& P, BlockCandT<CAP>& bc, TopkScratch& sc) {
    __syncthreads();
    if (bc.n == 0) return;   // uniform: almost every block
    if (P.k > 0) block_cut(bc, sc, P.k);
    block_flush(P, bc);
}

// ---------------------------------------------------------------------------
// Global selection and Ehrenfests' step, run by one block: the last block of
// a stream-collide launch, or the stand-alone select kernel.
//   mode 0: select among the candidates (or replay a given list), overwrite
//           the LBGK output of the selected sites with f* (Sec. 3.2; (ESLB)),
//           log the count and advance the step counter;
//   mode 1: select only (the select-only test hook; and a slab's own k best,
//           with their keys, when the global selection is made across
//           slabs).
// Candidates are staged in shared memory when they fit; larger sets are
// ranked in place in global memory.
// ---------------------------------------------------------------------------
struct SelectShared {
    TopkScratch sc;
    unsigned cnt;
};

// The Ehrenfests' step at one site: g, its post-collision populations in,
// f* out (not yet rounded as the storage holds it).  The collision conserves
// every moment f* depends on, so this is f* of the pre-collision state.
template <typename L, typename S, int EQ>
__device__ __forceinline__ void ehrenfest_value(const Params& P, typename Store<S>::T* g) {
    using T = typename Store<S>::T;
    T gs[L::Q], rho, ux, uy;
    site_equilibrium<L, T, EQ>(P, g, gs, rho, ux, uy);
    if constexpr (Store<S>::kProject) {
        // f' = f* = f - (f - f*), with the conserved moments of
        // f - f* freed of rounding as in the collision
        T d[L::Q];
#pragma unroll
        for (int i = 0; i < L::Q; i++) d[i] = g[i] - gs[i];
        conserve_neq<L, EQ>(d);
#pragma unroll
        for (int i = 0; i < L::Q; i++) gs[i] = g[i] - d[i];
    }
#pragma unroll
    for (int i = 0; i < L::Q; i++) g[i] = gs[i];
}
template <typename L, typename S, int EQ>
__device__ __forceinline__ void ehrenfest_site(const Params& P, long long o, typename Store<S>::T* g) {
    ehrenfest_value<L, S, EQ>(P, g);
#pragma unroll
    for (int i = 0; i < L::Q; i++) Store<S>::store(P.dst, i * P.plane + o, store_round<L, S>(i, g[i]));
}

constexpr int kRankMax = 256;   // candidates ranked by counting, one per thread

// What bounds this: one block runs it while the rest of the GPU is done, a
// chain of dependent loads.  Up to kRankMax candidates (and no more than the
// block has threads) go one per thread: a candidate's rank is the number of
// candidates before it in the selection's total order, counted in shared
// memory, its site's populations are fetched meanwhile, and the threads of
// rank below k perform the Ehrenfests' step at once -- one load after
// another: count, candidate, populations.  The radix select that larger sets
// take costs several block barriers and passes and puts its result in global
// memory first: from the ticket to the last store 6 us against 4 us on the
// 4096 x 2048 cylinder.
template <typename L, typename S, int EQ>
__device__ __noinline__ void select_and_fix(const Params& P, SelectShared& ss,
                                            unsigned long long* stage_key, unsigned* stage_idx,
                                            int stage_cap, int mode) {
    using T = typename Store<S>::T;
    const int tid = threadIdx.x, nt = blockDim.x;
    const long long t = __ldcg(P.step);   // used at the end: its latency overlaps the selection
    long long r = 0;
    bool replay = false;
    if (P.replay_cnt) {
        r = t - P.replay_t0;
        replay = r >= 0 && r < P.replay_n;
    }
    const int n = P.k > 0 && !replay ? (int)__ldcg(P.cand_count) : 0;
    int m;   // sites selected
    if (!replay && n <= min(min(nt, kRankMax), stage_cap)) {
        unsigned long long key = 0ull;
        unsigned id = 0u;
        T g[L::Q];
        long long o = 0;
        if (tid < n) {
            id = __ldcg(P.cand_idx + tid);
            key = __ldcg(P.cand_key + tid);
            stage_key[tid] = key;
            stage_idx[tid] = id;
            if (mode == 0) {
                o = (long long)(id / (unsigned)P.nx) * P.nxp + id % (unsigned)P.nx;
#pragma unroll
                for (int i = 0; i < L::Q; i++) g[i] = Store<S>::load(P.dst, i * P.plane + o);
            }
        }
        __syncthreads();
        if (tid < n) {
            int rank = tid;
            if (n > P.k) {
                rank = 0;
#pragma unroll 8
                for (int e = 0; e < n; e++) {
                    const unsigned long long ke = stage_key[e];
                    rank += ke > key || (ke == key && stage_idx[e] < id);
                }
            }
            if (rank < P.k) {
                P.sel_idx[rank] = (int)id;
                if (P.sel_key) P.sel_key[rank] = key;
                if (mode == 0) ehrenfest_site<L, S, EQ>(P, o, g);
            }
        }
        m = min(n, P.k);
    } else {
        if (replay) {
            const int c = P.replay_cnt[r];
            const long long off = P.replay_off[r];
            for (int j = tid; j < c; j += nt) P.sel_idx[j] = P.replay_idx[off + j];
            m = c;
        } else if (n <= P.k) {
            for (int j = tid; j < n; j += nt) {
                P.sel_idx[j] = (int)__ldcg(P.cand_idx + j);
                if (P.sel_key) P.sel_key[j] = __ldcg(P.cand_key + j);
            }
            m = n;
        } else {
            const bool staged = n <= stage_cap;
            if (staged) {
                for (int j = tid; j < n; j += nt) {
                    stage_key[j] = __ldcg(P.cand_key + j);
                    stage_idx[j] = __ldcg(P.cand_idx + j);
                }
                __syncthreads();
            }
            auto keyat = [&](int e) { return staged ? stage_key[e] : __ldcg(P.cand_key + e); };
            auto idat = [&](int e) { return staged ? stage_idx[e] : __ldcg(P.cand_idx + e); };
            const Thresh th = block_topk(ss.sc, n, P.k, keyat, idat);
            if (tid == 0) ss.cnt = 0;
            __syncthreads();
            for (int j = tid; j < n; j += nt) {
                const unsigned id = idat(j);
                const unsigned long long key = keyat(j);
                if (th.selected(key, id)) {
                    const unsigned s = atomicAdd(&ss.cnt, 1u);
                    if (s < (unsigned)P.k) {   // exactly k; bounds the write
                        P.sel_idx[s] = (int)id;
                        if (P.sel_key) P.sel_key[s] = key;
                    }
                }
            }
            m = P.k;
        }
        __syncthreads();
        if (mode == 0) {
            const long long nsites = (long long)P.nx * P.ny;
            for (int j = tid; j < m; j += nt) {
                const int site = P.sel_idx[j];
                if (site < 0 || site >= nsites) { atomicOr(P.err, ERR_REPLAY); continue; }
                const int x = site % P.nx, y = site / P.nx;
                if (is_solid(P, x, y)) { atomicOr(P.err, ERR_REPLAY); continue; }
                const long long o = (long long)y * P.nxp + x;
                T g[L::Q];
#pragma unroll
                for (int i = 0; i < L::Q; i++) g[i] = Store<S>::load(P.dst, i * P.plane + o);
                ehrenfest_site<L, S, EQ>(P, o, g);
            }
        }
        __syncthreads();
    }
    if (tid == 0) {
        // (every thread has read the count: the barriers above)
        *P.sel_count = m;
        *P.cand_count = 0;
        if (mode == 0) {
            P.count_ring[t % P.ring_cap] = m;
            *P.step = t + 1;
        }
    }
}

// End of a stream-collide block: publish the block's k best candidates and
// its writes and take a ticket; the block that takes the last ticket runs the
// global selection and the Ehrenfests' step for the whole grid.  No block
// ever waits for another.
template <typename L, typename S, int EQ, typename BC>
__device__ __forceinline__ void finish_parts(const Params& P, int& is_last, SelectShared& ss, BC& bc,
                                             unsigned long long* stage_key, unsigned* stage_idx,
                                             int stage_cap) {
    block_finish(P, bc, ss.sc);
    // the barrier makes the block's writes visible to thread 0, whose
    // device-scope fence then orders all of them before the ticket
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        const unsigned nb = gridDim.x * gridDim.y;
        const unsigned tk = atomicAdd(P.ticket, 1u);
        __threadfence();
        is_last = (tk == nb - 1);
    }
    __syncthreads();
    if (is_last) {
        __threadfence_block();
        select_and_fix<L, S, EQ>(P, ss, stage_key, stage_idx, stage_cap, P.slab ? 1 : 0);
        if (threadIdx.x == 0) {
            *P.ticket = 0;
            if (P.tile_counter) *P.tile_counter = 0;
        }
    }
}

// Shared state of the kernels whose sites come from registers.  CAP: room
// for a round of the block's sites above what a cut keeps.  p: the launch's
// parameters for the out-of-line paths.
template <int CAP>
struct SiteShared {
    Params p;
    SelectShared ss;
    unsigned long long key[kStage];
    unsigned idx[kStage];
    BlockCandT<CAP> bc;
    int is_last;
};

// Pre-collision deviations of a site by the boundary rules, out of line (the
// tiles without any keep their registers).
template <typename L, typename S>
__device__ __noinline__ PopArr<L::Q, typename Store<S>::T> gather_ruled(const Params& P, int x, int y) {
    PopArr<L::Q, typename Store<S>::T> a;
    gather_site<L, S>(P, x, y, a.v);
    return a;
}

// ---------------------------------------------------------------------------
// Vector loads and stores of VEC consecutive populations (aligned).  Ordinary
// loads throughout, and no __restrict__ on the source field: a kernel launched
// as a programmatic dependent is alive while its predecessor still writes the
// field it will read, so the read-only data path (__ldg) is not for it, and a
// read-only promise would let a load move above griddepcontrol.wait.
// ---------------------------------------------------------------------------
template <typename S, int VEC> struct VecIO;
template <typename S> struct VecIO<S, 1> {
    __device__ static void load(const void* p, long long i, typename Store<S>::T* v) {
        v[0] = Store<S>::load(p, i);
    }
    __device__ static void store(void* p, long long i, const typename Store<S>::T* v) {
        Store<S>::store(p, i, v[0]);
    }
};
template <> struct VecIO<float, 4> {
    __device__ static void load(const void* p, long long i, float* v) {
        const float4 a = *reinterpret_cast<const float4*>(static_cast<const float*>(p) + i);
        v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
    }
    __device__ static void store(void* p, long long i, const float* v) {
        *reinterpret_cast<float4*>(static_cast<float*>(p) + i) = make_float4(v[0], v[1], v[2], v[3]);
    }
};
template <> struct VecIO<float, 2> {
    __device__ static void load(const void* p, long long i, float* v) {
        const float2 a = *reinterpret_cast<const float2*>(static_cast<const float*>(p) + i);
        v[0] = a.x; v[1] = a.y;
    }
    __device__ static void store(void* p, long long i, const float* v) {
        *reinterpret_cast<float2*>(static_cast<float*>(p) + i) = make_float2(v[0], v[1]);
    }
};
template <> struct VecIO<double, 4> {
    __device__ static void load(const void* p, long long i, double* v) {
        const double2* q = reinterpret_cast<const double2*>(static_cast<const double*>(p) + i);
        const double2 a = q[0], b = q[1];
        v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;
    }
    __device__ static void store(void* p, long long i, const double* v) {
        double2* q = reinterpret_cast<double2*>(static_cast<double*>(p) + i);
        q[0] = make_double2(v[0], v[1]);
        q[1] = make_double2(v[2], v[3]);
    }
};
template <> struct VecIO<double, 2> {
    __device__ static void load(const void* p, long long i, double* v) {
        const double2 a = *reinterpret_cast<const double2*>(static_cast<const double*>(p) + i);
        v[0] = a.x; v[1] = a.y;
    }
    __device__ static void store(void* p, long long i, const double* v) {
        *reinterpret_cast<double2*>(static_cast<double*>(p) + i) = make_double2(v[0], v[1]);
    }
};
template <> struct VecIO<__half, 4> {
    __device__ static void load(const void* p, long long i, float* v) {
        const uint2 a = *reinterpret_cast<const uint2*>(static_cast<const __half*>(p) + i);
        const float2 lo = __half22float2(*reinterpret_cast<const __half2*>(&a.x));
        const float2 hi = __half22float2(*reinterpret_cast<const __half2*>(&a.y));
        v[0] = lo.x; v[1] = lo.y; v[2] = hi.x; v[3] = hi.y;
    }
    __device__ static void store(void* p, long long i, const float* v) {
        __half2 lo = __floats2half2_rn(v[0], v[1]);
        __half2 hi = __floats2half2_rn(v[2], v[3]);
        uint2 a;
        a.x = *reinterpret_cast<unsigned*>(&lo);
        a.y = *reinterpret_cast<unsigned*>(&hi);
        *reinterpret_cast<uint2*>(static_cast<__half*>(p) + i) = a;
    }
};
template <> struct VecIO<__half, 2> {
    __device__ static void load(const void* p, long long i, float* v) {
        const unsigned a = *reinterpret_cast<const unsigned*>(static_cast<const __half*>(p) + i);
        const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&a));
        v[0] = f.x; v[1] = f.y;
    }
    __device__ static void store(void* p, long long i, const float* v) {
        __half2 h = __floats2half2_rn(v[0], v[1]);
        *reinterpret_cast<unsigned*>(static_cast<__half*>(p) + i) = *reinterpret_cast<unsigned*>(&h);
    }
};

template <> struct VecIO<plain32, 4> {
    __device__ static void load(const void* p, long long i, float* v) { VecIO<float, 4>::load(p, i, v); }
    __device__ static void store(void* p, long long i, const float* v) { VecIO<float, 4>::store(p, i, v); }
};
template <> struct VecIO<plain32, 2> {
    __device__ static void load(const void* p, long long i, float* v) { VecIO<float, 2>::load(p, i, v); }
    __device__ static void store(void* p, long long i, const float* v) { VecIO<float, 2>::store(p, i, v); }
};

// Two adjacent populations (columns c, c + 1 with c even: 8-byte aligned
// for FP32, 4-byte for FP16, 16-byte for FP64) of a staged plane row or of
// a population plane, loaded or stored with one access.
template <typename S> struct PairIO;
template <> struct PairIO<float> {
    __device__ static void load(const float* p, float& a, float& b) {
        const float2 v = *reinterpret_cast<const float2*>(p);
        a = v.x;
        b = v.y;
    }
    __device__ static void store(float* p, float a, float b) { *reinterpret_cast<float2*>(p) = make_float2(a, b); }
};
template <> struct PairIO<plain32> {
    __device__ static void load(const plain32* p, float& a, float& b) {
        PairIO<float>::load(reinterpret_cast<const float*>(p), a, b);
    }
    __device__ static void store(plain32* p, float a, float b) {
        PairIO<float>::store(reinterpret_cast<float*>(p), a, b);
    }
};
template <> struct PairIO<__half> {
    __device__ static void load(const __half* p, float& a, float& b) {
        const float2 v = __half22float2(*reinterpret_cast<const __half2*>(p));
        a = v.x;
        b = v.y;
    }
    __device__ static void store(__half* p, float a, float b) {
        *reinterpret_cast<__half2*>(p) = __floats2half2_rn(a, b);
    }
};
template <> struct PairIO<double> {
    __device__ static void load(const double* p, double& a, double& b) {
        const double2 v = *reinterpret_cast<const double2*>(p);
        a = v.x;
        b = v.y;
    }
    __device__ static void store(double* p, double a, double b) {
        *reinterpret_cast<double2*>(p) = make_double2(a, b);
    }
};

// Interior-path accessors with 32-bit element indices (every population
// array holds fewer than 2^31 elements; checked at creation).
template <typename S, int VEC>
__device__ __forceinline__ void load_vec(const S* p, int i, typename Store<S>::T* v) {
    VecIO<S, VEC>::load(p + i, 0, v);
}
template <typename S, int VEC>
__device__ __forceinline__ void store_vec(S* __restrict__ p, int i, const typename Store<S>::T* v) {
    VecIO<S, VEC>::store(p + i, 0, v);
}

// A row tile [x0, x0 + TX) of row y is interior when the tile and its
// one-site halo are fluid and inside the grid: its gather is a pure shift.
template <int TX>
__device__ __forceinline__ bool tile_interior(const Params& P, int x0, int y) {
    if (x0 < 1 || x0 + TX > P.nx - 1 || y < 1 || y > P.ny - 2) return false;
    if (P.ow > 0) {
        const bool apart = (x0 + TX + 1 <= P.ox0) || (x0 - 1 >= P.ox0 + P.ow) ||
                           (y + 2 <= P.oy0) || (y - 1 >= P.oy0 + P.oh);
        if (!apart) return false;
    }
    return true;
}

// ---------------------------------------------------------------------------
// K1 for D2Q9, persistent: the grid holds as many blocks as fit on the
// GPU at once; each block processes a contiguous range of row tiles of
// 32 x VEC consecutive sites, its warps taking the range's tiles in turn.
// Interior tiles: aligned VEC-wide loads per population plane, the
// x-shifted planes completed by one warp shuffle and one halo load.
// Boundary tiles (and the first step after a state upload): per-site gather
// with the boundary rules (out of line), then the same update.
// For grids of one or two tiles per warp: bound by the chain launch - loads -
// update - selection.  So the launch overlaps the previous step's end, a
// boundary tile costs one more gather and no update code of its own, and the
// sites the dS bound does not clear are resolved after their tile instead of
// in a pass of the whole block at the end.  600 x 500, FP32, one run alone:
// 16.1 -> 13.4 us per step (three side by side: 7.8 us each, as before).
// ---------------------------------------------------------------------------
template <typename S, int EQ, int VEC, int WARPS, int MINB>
__global__ void __launch_bounds__(32 * WARPS, MINB) k_collide_d2q9(const __grid_constant__ Params P) {
    using L = D2Q9;
    using T = typename Store<S>::T;
    constexpr int TX = 32 * VEC;
    constexpr int kRound = TX * WARPS;             // sites of a round (one tile per warp)
    constexpr int kCap = kRound + kBlockCand;
    __shared__ SiteShared<kCap> sh;
    __shared__ MlpSlot<EQ> mslot;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) {
        sh.p = P;
        sh.bc.n = 0;
    }
    // Each block owns a contiguous range of row tiles (row-major); its warps
    // take the range's tiles in turn.  Boundary tiles, which cost more, are
    // then spread evenly over blocks.
    const int tiles_x = (P.nx + TX - 1) / TX;
    const int tiles = tiles_x * P.ny;
    const int per_block = (tiles + gridDim.x - 1) / gridDim.x;
    const int t0 = blockIdx.x * per_block;
    const int t1 = min(t0 + per_block, tiles);
    const int rounds = t1 > t0 ? (t1 - t0 + WARPS - 1) / WARPS : 0;
    int y = (t0 + warp) / tiles_x, xt = t0 + warp - y * tiles_x;
    // a programmatic dependent of the previous kernel in the stream, as the
    // staged kernel: nothing above reads device memory a kernel writes
    asm volatile("griddepcontrol.wait;" ::: "memory");
    mslot.fill(P);
    __syncthreads();
    const long long t = P.probe_ring ? __ldcg(P.step) : 0;   // (the probe's log only)
    const S* src = static_cast<const S*>(P.src);
    S* __restrict__ dst = static_cast<S*>(P.dst);
    const int nxp = P.nxp, plane = (int)P.plane;
    bool nonfinite = false;
    NewtonCount nc = {0, 0, 0, 0};
    // candidates appended by the warp since the block's last cut; the block
    // cuts (or flushes) once some warp used more than its share of the room
    // above what a cut keeps, so that the next round fits
    unsigned count = 0u;
    const int kept = P.k > 0 && P.k < kBlockCand ? P.k : 0;
    const unsigned share = (unsigned)((kBlockCand - kept) / WARPS);
    for (int r = 0; r < rounds; r++) {
        if (t0 + r * WARPS + warp < t1) {
            const int x0 = xt * TX;
            const int xs = x0 + lane * VEC;
            const int row = y * nxp + xs;
            const bool interior = !P.prestream && tile_interior<TX>(P, x0, y);
            T g[VEC][L::Q];
            unsigned fluid = (1u << VEC) - 1u;
            if (interior) {
#pragma unroll
                for (int i = 0; i < L::Q; i++) {
                    const int at = i * plane + row - L::cy(i) * nxp;
                    T v[VEC];
                    load_vec<S, VEC>(src, at, v);
                    if (L::cx(i) == 0) {
#pragma unroll
                        for (int s = 0; s < VEC; s++) g[s][i] = v[s];
                    } else if (L::cx(i) == 1) {
                        // source x - 1: the previous lane's last element
                        T prev = __shfl_up_sync(0xffffffffu, v[VEC - 1], 1);
                        if (lane == 0) prev = Store<S>::load(src + at - 1, 0);
                        g[0][i] = prev;
#pragma unroll
                        for (int s = 1; s < VEC; s++) g[s][i] = v[s - 1];
                    } else {
                        // source x + 1: the next lane's first element
                        T next = __shfl_down_sync(0xffffffffu, v[0], 1);
                        if (lane == 31) next = Store<S>::load(src + at + VEC, 0);
#pragma unroll
                        for (int s = 0; s < VEC - 1; s++) g[s][i] = v[s + 1];
                        g[VEC - 1][i] = next;
                    }
                }
            } else {
#pragma unroll
                for (int s = 0; s < VEC; s++) {
                    const int x = xs + s;
                    if (x < P.nx && !is_solid(P, x, y)) {
                        const auto a = gather_ruled<L, S>(sh.p, x, y);
#pragma unroll
                        for (int i = 0; i < L::Q; i++) g[s][i] = a.v[i];
                    } else {
                        // no site of the run (solid sites hold zeros in both
                        // buffers from the start): the rest state at unit
                        // density, not stored, never pending
                        fluid &= ~(1u << s);
#pragma unroll
                        for (int i = 0; i < L::Q; i++) g[s][i] = T(L::w(i)) * (T(1) - Par<T>::rho0(P));
                    }
                }
                __syncwarp();
            }
            unsigned pend = 0u;
#pragma unroll
            for (int s = 0; s < VEC; s++) {
                NewtonCount one = nc;
                float mu3 = 0.0f;
                if constexpr (EQ == EQ_ENERGY_MLP) mu3 = mlp_site_start<T>(P, mslot.s, true, g[s]);
                const bool p = update_site<L, T, EQ, Store<S>::kProject>(P, g[s], (fluid >> s) & 1u ? xs + s : -2, y, t,
                                                                         nonfinite, one, mu3);
                if ((fluid >> s) & 1u) {
                    nc = one;
                    if (p) pend |= 1u << s;
                }
            }
            if (interior) {
#pragma unroll
                for (int i = 0; i < L::Q; i++) {
                    T v[VEC];
#pragma unroll
                    for (int s = 0; s < VEC; s++) v[s] = store_round<L, S>(i, g[s][i]);
                    store_vec<S, VEC>(dst, i * plane + row, v);
                }
            } else {
#pragma unroll
                for (int s = 0; s < VEC; s++)
                    if ((fluid >> s) & 1u) {
#pragma unroll
                        for (int i = 0; i < L::Q; i++)
                            Store<S>::store(dst + i * plane + row + s, 0, store_round<L, S>(i, g[s][i]));
                    }
            }
            // the tile's pending sites, gathered again (from L2)
            if (__any_sync(0xffffffffu, pend != 0u)) {
#pragma unroll 1
                for (int s = 0; s < VEC; s++) {
                    T ds = T(-1);
                    if ((pend >> s) & 1u) ds = resolve_ds<L, S, EQ>(sh.p, xs + s, y);
                    count += block_push<T>(P, sh.bc, ds > Par<T>::delta(P), ds, (unsigned)(y * P.nx + xs + s));
                }
            }
            xt += WARPS;
            while (xt >= tiles_x) { xt -= tiles_x; y++; }
        }
        if (r + 1 < rounds && __syncthreads_or(count > share)) {
            if (P.k < kBlockCand) block_cut(sh.bc, sh.ss.sc, P.k);
            else block_flush(sh.p, sh.bc);
            count = 0u;
        }
    }
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (nonfinite) atomicOr(P.err, ERR_NONFINITE);
    if constexpr (EQ >= EQ_ENERGY) flush_newton(P, nc);
    finish_parts<L, S, EQ>(sh.p, sh.is_last, sh.ss, sh.bc, sh.key, sh.idx, kStage);
}

// ---------------------------------------------------------------------------
// K1 for D2Q9 with tiles staged in shared memory by the tensor memory
// accelerator.  A block tile is R rows x 128 sites.  Population i at row y
// comes from row y - v_iy of the source field, so for each of the 9 planes
// one 3-D bulk tensor copy brings exactly the R rows y0 - v_iy ..
// y0 - v_iy + R - 1 the tile pulls from that plane, over columns x0 - H ..
// x0 + 128 + H (H elements = 16 bytes on each side, which keeps every copy
// 16-byte aligned).  Copies complete on an mbarrier; STAGES tiles are in
// flight per block, so the bytes in flight do not depend on registers.
// Warp w computes row w of the tile, lane l the site pairs x0 + 2 l + 64 s,
// + 1: shared-memory reads and global stores are both consecutive across the
// warp.  In rows at the y sides or the obstacle, patch_row first writes what
// the boundary rules replace into the staged planes; the x = 0 and
// x = nx - 1 columns are edge items of their own.  Every wait on an
// mbarrier is bounded: on expiry the block flags ERR_TIMEOUT, stops issuing
// copies, waits (bounded) for the copies it issued, and ends.
// ---------------------------------------------------------------------------
constexpr int kTmaTX = 128;
constexpr long long kWaitLimit = 1ll << 22;   // try_wait polls before a wait is declared failed

__device__ __forceinline__ unsigned smem_u32(const void* p) {
    return (unsigned)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void mbar_init(unsigned long long* bar, unsigned count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(unsigned long long* bar, unsigned bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
                 "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(unsigned long long* bar, unsigned parity) {
    unsigned ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
// bounded wait; false when the limit expired
__device__ __forceinline__ bool mbar_wait(unsigned long long* bar, unsigned parity) {
    for (long long it = 0; it < kWaitLimit; it++)
        if (mbar_try_wait(bar, parity)) return true;
    return false;
}
// The same for a whole warp (every lane calls): false on every lane when any
// lane's wait gave up, so that the warp leaves, or goes on, as one.
__device__ __forceinline__ bool warp_wait(unsigned long long* bar, unsigned parity) {
    return __all_sync(0xffffffffu, mbar_wait(bar, parity));
}
__device__ __forceinline__ void tma_load_3d(void* dst, const CUtensorMap* tm, int c0, int c1, int c2,
                                            unsigned long long* bar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(smem_u32(dst)),
        "l"(reinterpret_cast<unsigned long long>(tm)), "r"(c0), "r"(c1), "r"(c2), "r"(smem_u32(bar))
        : "memory");
}

template <typename S, int R, int TX = kTmaTX>
struct TmaLayout {
    static constexpr int H = 16 / (int)sizeof(S);          // halo columns (16 bytes)
    static constexpr int W = TX + 2 * H;                   // staged row length
    static constexpr int ROWS = R;                         // plane i: rows y0 - v_iy .. y0 - v_iy + R - 1
    static constexpr int BOX_BYTES = ROWS * W * (int)sizeof(S);
    static constexpr int PLANE_BYTES = (BOX_BYTES + 127) / 128 * 128;   // 128-byte aligned boxes
    static constexpr int PLANE = PLANE_BYTES / (int)sizeof(S);
    static constexpr int STAGE_BYTES = 9 * PLANE_BYTES;
    static constexpr int TX_BYTES = 9 * BOX_BYTES;         // bytes one tile's copies deliver
};

// Candidate buffer of a staged block: room for one tile's sites above what
// a cut keeps (the block cuts between tiles; the global list, which has a
// slot per site, takes what a tile begun before a cut finds no room for).
template <int R, int TX>
constexpr int tma_cand_cap() {
    return TX * R + kBlockCand;
}

// The stages of a staged block, handed on without a barrier of the block: a
// warp that has finished with a stage's tile says so (done), and the one that
// finishes last refills the stage at once with the work thread 0 has claimed
// for it (next).  A warp therefore never waits for the others, only for its
// next tile's copies, and every stage but those being computed is in flight.
// With one barrier per tile instead (every warp waiting for the slowest, one
// stage idle), barriers were the largest stall (FP16: 2.6 of 11 cycles per
// issue, now 0.5).  us per step, exports shared out, before and now: 4096 x
// 2048 polynomial FP32 96.9, 94.1; FP16 71.2, 70.3; 2048 x 1024 FP64 300,
// 289; ELBM 56.2, 55.1; energy 49.9, 48.7; 64 runs in one launch 431, 421.
template <int N>
struct StageRing {
    int tile[N];   // work a stage holds (-1: none left; -2 - e: edge item e)
    int x0[N], y0[N];   // the tile's origin
    int next[N];   // work for the stage's next refill
    int done[N];   // warps that have finished with the stage's work
};

// The calling warp has finished with a stage (lane 0 calls, after a
// __syncwarp): true for the last of n warps, which sees the others' accesses
// as done and refills the stage.
__device__ __forceinline__ bool stage_leave(int* done, int n) {
    int before;
    asm volatile("atom.acq_rel.cta.shared::cta.add.u32 %0, [%1], 1;" : "=r"(before) : "r"(smem_u32(done)) : "memory");
    if (before != n - 1) return false;
    *done = 0;
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    return true;
}

// Shared state of a staged block besides its tiles.  p: the launch's
// parameters, for the out-of-line paths (a reference to the kernel's
// __grid_constant__ parameter passed to a function that is not inlined
// reads it through generic loads of the parameter space; the shared copy
// answers at shared-memory latency).
constexpr unsigned kCutAsked = 0x80000000u, kGaveUp = 0xffffffffu;
template <int CAP>
struct TmaShared {
    Params p;
    SelectShared ss;
    BlockCandT<CAP> bc;
    int is_last;
    int abort;
    unsigned begun;   // the last work any warp has begun (its ordinal); kCutAsked: cut before the next
    unsigned met;     // outcome of the warps' rendezvous before a cut (rendezvous_met)
    StageRing<8> ring;
};

template <typename S, int R, int STAGES, int EQ, int TX = kTmaTX>
constexpr size_t tma_smem_bytes() {
    return 128 + (size_t)STAGES * TmaLayout<S, R, TX>::STAGE_BYTES + 8 * (STAGES + 1) +
           sizeof(TmaShared<tma_cand_cap<R, TX>()>) + 16 +
           (EQ == EQ_ENERGY_MLP ? sizeof(MlpSlot<EQ>) + 16 : 0);
}

// Where a staged tile's candidates go (put: every lane of the warp calls,
// with its site's dS, -1 for a site the dS bound cleared; the sites the
// bound does not clear have their exact dS evaluated on the tile, from the
// staged planes or in the update).  CandSink: the block's buffer.
// GlobalCandSink: the run's global list (a kernel whose tiles belong to
// different runs).
template <int CAP>
struct CandSink {
    BlockCandT<CAP>* bc;
    template <typename T>
    __device__ __forceinline__ void put(const Params& P, T ds, unsigned site) {
        block_push<T>(P, *bc, ds > Par<T>::delta(P), ds, site);
    }
};
struct GlobalCandSink {
    template <typename T>
    __device__ __forceinline__ void put(const Params& P, T ds, unsigned site) {
        warp_push<T>(P, ds > Par<T>::delta(P), ds, site);
    }
};

// What a warp carries from tile to tile; passed to and returned from the
// out-of-line paths by value, so that it stays in registers.
template <typename Sink>
struct TileState {
    Sink sink;
    NewtonCount nc;
    bool nonfinite;
};

// Pre-collision deviations of site (x, y) of a staged tile: the same rules
// as gather_site (free flight, Sec. 4.2 boundaries).  Plane j's window holds
// source rows y0 - v_jy .. y0 - v_jy + R - 1 (box[j][row][col] with
// row = sy - y0 + v_jy, col = sx - x0 + H); a rule that reads a plane
// outside its window (a bounce-back or a mirror at the tile's edge rows, the
// outlet column) reads the source field instead.  Not used with periodic
// sides, nor for the first step after a state upload.
template <typename S, int R, int TX = kTmaTX>
__device__ __forceinline__ void gather_site_smem(const Params& P, const S* box, int x0, int y0, int x,
                                                 int y, typename Store<S>::T* g) {
    using L = D2Q9;
    using T = typename Store<S>::T;
    using LY = TmaLayout<S, R, TX>;
    auto at = [&](int j, int sx, int sy) {
        const int r = sy - y0 + L::cy(j), c = sx - x0 + LY::H;
        if ((unsigned)r < (unsigned)R && (unsigned)c < (unsigned)LY::W)
            return Store<S>::load(box + j * LY::PLANE + r * LY::W + c, 0);
        return Store<S>::load(P.src, j * P.plane + (long long)sy * P.nxp + sx);
    };
    bool have_out = false;
    unsigned wall_mask = 0u;
    T gout[L::Q];
#pragma unroll
    for (int i = 0; i < L::Q; i++) {
        const int cx = L::cx(i), cy = L::cy(i);
        int sx = x - cx;
        const int sy = y - cy;
        if (sx < 0 || sx >= P.nx) {
            const int kind = sx < 0 ? P.bc[0] : P.bc[1];
            if (kind == BC_OUTLET_COPY) {
                sx = x;   // the column beyond the side is a copy of the side column
            } else if (kind == BC_INLET) {
                g[i] = (T)P.gin[i];
            } else if (kind == BC_OUTLET) {
                if (!have_out) {
                    T v[L::Q];
#pragma unroll
                    for (int j = 0; j < L::Q; j++) v[j] = at(j, P.nx - 2, y);
                    outlet_equilibrium<L, T>(P, v, gout);
#pragma unroll
                    for (int j = 0; j < L::Q; j++) gout[j] = store_round<L, S>(j, gout[j]);
                    have_out = true;
                }
                g[i] = gout[i];
            } else {
                g[i] = at(L::opp(i), x, y);
            }
            if (kind != BC_OUTLET_COPY) continue;
        }
        if (sy < 0 || sy >= P.ny) {
            const int kind = sy < 0 ? P.bc[2] : P.bc[3];
            g[i] = kind == BC_FREESLIP ? at(L::mir_y(i), sx, y) : at(L::opp(i), x, y);
            continue;
        }
        if (is_solid(P, sx, sy)) {
            g[i] = at(L::opp(i), x, y);
            if (P.wall == WALL_DIFFUSE) wall_mask |= 1u << i;
        } else {
            g[i] = at(i, sx, sy);
        }
    }
    if (wall_mask) diffuse_wall<L, T>(wall_mask, g);
}

// The sites of a staged row next to a diffuse wall in FP16 storage, one by
// one with the boundary rules: the wall's populations are FP32 values that a
// staged FP16 row cannot hold (patch_row serves every other case).  Out of
// line, so that the interior path is allocated registers on its own.
template <typename S, int EQ, int R, int TX, typename Sink>
__device__ __noinline__ TileState<Sink> tma_tile_general(const Params& P, const S* box, int x0, int y0, long long t,
                                                         TileState<Sink> state, MlpSlot<EQ>& mslot) {
    using L = D2Q9;
    using T = typename Store<S>::T;
    using LY = TmaLayout<S, R, TX>;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    S* __restrict__ dst = static_cast<S*>(P.dst);
    const int nxp = P.nxp, plane = (int)P.plane;
    const bool periodic = P.bc[0] == BC_PERIODIC || P.bc[2] == BC_PERIODIC;
    const int y = y0 + warp;
    const S* sb = box + warp * LY::W + LY::H;
#pragma unroll 1
    for (int s = 0; s < TX / 32; s++) {
        const int x = x0 + lane + 32 * s;
        T ds = T(-1);
        // the learned form enters with every lane (its warm start is a
        // warp-wide evaluation); lanes outside the grid then carry no site
        // the columns x = 0 and x = nx - 1 are updated apart (edge_item)
        const bool mine = x < P.nx && y < P.ny && !(x == 0 || x == P.nx - 1);
        if (EQ == EQ_ENERGY_MLP || mine) {
            const bool inside = mine;
            const int c = x - x0;
            const int o = y * nxp + x;
            const bool near_obstacle = P.ow > 0 && x >= P.ox0 - 1 && x <= P.ox0 + P.ow &&
                                       y >= P.oy0 - 1 && y <= P.oy0 + P.oh;
            const bool shift = x >= 1 && x <= P.nx - 2 && y >= 1 && y <= P.ny - 2 && !near_obstacle;
            T g[L::Q];
            bool fluid = inside;
            if (!inside) {
#pragma unroll
                for (int i = 0; i < L::Q; i++) g[i] = T(0);
            } else if (shift) {
#pragma unroll
                for (int i = 0; i < L::Q; i++) g[i] = Store<S>::load(sb + i * LY::PLANE + c - L::cx(i), 0);
            } else if (is_solid(P, x, y)) {
                fluid = false;
#pragma unroll
                for (int i = 0; i < L::Q; i++) g[i] = T(0);
            } else if (periodic) {
                gather_site<L, S>(P, x, y, g);
            } else {
                gather_site_smem<S, R, TX>(P, box, x0, y0, x, y, g);
            }
            float mu3 = 0.0f;
            if constexpr (EQ == EQ_ENERGY_MLP) {
                __syncwarp();
                mu3 = mlp_site_start<T>(P, mslot.s, fluid, g);
            }
            if (fluid)
                update_site<L, T, EQ, Store<S>::kProject, true, true>(P, g, x, y, t, state.nonfinite, state.nc, mu3,
                                                                      &ds);
            if (inside) {
#pragma unroll
                for (int i = 0; i < L::Q; i++)
                    Store<S>::store(dst + i * plane + o, 0, fluid ? store_round<L, S>(i, g[i]) : g[i]);
            }
        }
        state.sink.put(P, ds, (unsigned)(y * P.nx + x));
    }
    return state;
}


// The columns x = 0 and x = nx - 1 of the grid (the sites whose sources
// leave the grid in x), apart from the staged tiles: edge item e covers
// sites e * 32 R .. (e + 1) * 32 R - 1 of the list x = 0 (rows 0 .. ny - 1)
// then x = nx - 1, one site per lane, gathered from the source field with
// the boundary rules (gather_site).  Every lane of the block calls.
template <typename S, int EQ, int R, typename Sink>
__device__ __noinline__ TileState<Sink> edge_item(const Params& P, int item, long long t, TileState<Sink> state,
                                                  MlpSlot<EQ>& mslot) {
    using L = D2Q9;
    using T = typename Store<S>::T;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int ncols = P.nx > 1 ? 2 : 1;
    const int e = (item * R + warp) * 32 + lane;
    const bool inside = e < ncols * P.ny;
    const int x = inside && e >= P.ny ? P.nx - 1 : 0;
    const int y = inside ? (e >= P.ny ? e - P.ny : e) : 0;
    const bool fluid = inside && !is_solid(P, x, y);
    T g[L::Q];
    if (fluid) {
        gather_site<L, S>(P, x, y, g);
    } else {
#pragma unroll
        for (int i = 0; i < L::Q; i++) g[i] = T(0);
    }
    T ds = T(-1);
    float mu3 = 0.0f;
    if constexpr (EQ == EQ_ENERGY_MLP) mu3 = mlp_site_start<T>(P, mslot.s, fluid, g);
    if (fluid)
        update_site<L, T, EQ, Store<S>::kProject, true, true>(P, g, x, y, t, state.nonfinite, state.nc, mu3, &ds);
    if (inside) {
        S* dst = static_cast<S*>(P.dst);
        const long long o = (long long)y * P.nxp + x;
#pragma unroll
        for (int i = 0; i < L::Q; i++)
            Store<S>::store(dst, i * P.plane + o, fluid ? store_round<L, S>(i, g[i]) : g[i]);
    }
    state.sink.put(P, ds, (unsigned)(y * P.nx + x));
    return state;
}

// Exact dS of the pending sites of a clean staged row (warp w: row y; lane
// l: bit 2 s + h of pmask for column x0 + 2 l + 64 s + h), from the staged
// planes (the same values the update read) and f* recomputed as the update
// computed it; the sites go to the sink (which keeps the candidates).  Every
// lane of the warp calls.
template <typename S, int EQ, int R, int TX, typename Sink>
__device__ __noinline__ Sink resolve_staged_row(const Params& P, const S* box, int x0, int y, unsigned pmask,
                                                Sink sink) {
    using L = D2Q9;
    using T = typename Store<S>::T;
    using LY = TmaLayout<S, R, TX>;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const S* sb = box + warp * LY::W + LY::H;
#pragma unroll 1
    for (int b = 0; b < TX / 32; b++) {
        const int c = 2 * lane + 64 * (b >> 1) + (b & 1);
        T ds = T(-1);
        if ((pmask >> b) & 1u) {
            T g[L::Q], gs[L::Q], rho, ux, uy;
#pragma unroll
            for (int i = 0; i < L::Q; i++) g[i] = Store<S>::load(sb + i * LY::PLANE + c - L::cx(i), 0);
            site_equilibrium<L, T, EQ>(P, g, gs, rho, ux, uy);
            if (!ghost_column(P, x0 + c)) ds = site_ds<L, T, EQ>(P, g, gs);
        }
        sink.put(P, ds, (unsigned)(y * P.nx + x0 + c));
    }
    return sink;
}

// Boundary rules of a staged row, written into the staged planes: where the
// source of population i at a fluid site x of row y lies outside the grid in
// y or inside the obstacle, the staged slot it would be read from -- plane
// i, column x - v_ix of the warp's own row of that plane's window, which no
// other site reads -- takes the population the rule gives (gather_site; the
// columns x = 0 and x = nx - 1 go apart, edge_item).  The row then takes the
// interior path as it stands.  prestream (the first step after a state
// upload): every slot takes its own site's population.  The window rows
// outside the grid and the obstacle's sites hold zeros before.  Warp w: row
// y; every lane calls.
// Every load of a rule is issued before its first use, and whole rows at
// once at the y sides, so a patched row costs about one memory latency more
// than a plain one; evaluated site by site with the rules (the former path for
// every tile that touched a wall, the obstacle, a ragged edge or the probe) a
// row took about 10 us: at 2048 x 1024 the last block ended 12 - 28 us after
// the median one.
template <typename S, int R, int TX>
__device__ __noinline__ void patch_row(const Params& P, S* box, int x0, int y) {
    using L = D2Q9;
    using T = typename Store<S>::T;
    using LY = TmaLayout<S, R, TX>;
    constexpr int C = TX / 32;   // sites per lane
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    S* sb = box + warp * LY::W + LY::H;
    const S* src = static_cast<const S*>(P.src);
    const long long row = (long long)y * P.nxp;
    if (P.prestream) {
#pragma unroll 1
        for (int c = lane; c < TX; c += 32) {
            const int x = x0 + c;
            if (x < 1 || x > P.nx - 2) continue;
            S v[L::Q];
#pragma unroll
            for (int i = 0; i < L::Q; i++) v[i] = src[i * P.plane + row + x];
#pragma unroll
            for (int i = 0; i < L::Q; i++) sb[i * LY::PLANE + c - L::cx(i)] = v[i];
        }
    } else if (y == 0 || y == P.ny - 1) {
        // the three populations that come from beyond the side: v_y = e
        const int e = y == 0 ? 1 : -1;
        const int kind = P.bc[y == 0 ? 2 : 3];
        const long long far = (long long)(P.ny - 1 - y) * P.nxp;   // periodic: the opposite row
        S v[3][C];
#pragma unroll
        for (int p = 0; p < 3; p++) {
            const int cx = p == 0 ? 0 : (p == 1 ? 1 : -1);
            const int i = e > 0 ? (p == 0 ? 2 : (p == 1 ? 5 : 6)) : (p == 0 ? 4 : (p == 1 ? 8 : 7));
            const int mir = e > 0 ? (p == 0 ? 4 : (p == 1 ? 8 : 7)) : (p == 0 ? 2 : (p == 1 ? 5 : 6));
            const int opp = e > 0 ? (p == 0 ? 4 : (p == 1 ? 7 : 8)) : (p == 0 ? 2 : (p == 1 ? 6 : 5));
            const bool bb = kind != BC_PERIODIC && kind != BC_FREESLIP;
            const S* q = src + (kind == BC_PERIODIC ? i : (bb ? opp : mir)) * P.plane +
                         (kind == BC_PERIODIC ? far : row) + x0 - (bb ? 0 : cx);
#pragma unroll
            for (int s = 0; s < C; s++) {
                const int c = lane + 32 * s, x = x0 + c;
                if (x >= 1 && x <= P.nx - 2) v[p][s] = q[c];
            }
        }
#pragma unroll
        for (int p = 0; p < 3; p++) {
            const int cx = p == 0 ? 0 : (p == 1 ? 1 : -1);
            const int i = e > 0 ? (p == 0 ? 2 : (p == 1 ? 5 : 6)) : (p == 0 ? 4 : (p == 1 ? 8 : 7));
#pragma unroll
            for (int s = 0; s < C; s++) {
                const int c = lane + 32 * s, x = x0 + c;
                if (x >= 1 && x <= P.nx - 2) sb[i * LY::PLANE + c - cx] = v[p][s];
            }
        }
    }
    if (!P.prestream && P.ow > 0 && y >= P.oy0 - 1 && y <= P.oy0 + P.oh) {
#pragma unroll 1
        for (int c = lane; c < TX; c += 32) {
            const int x = x0 + c;
            const bool mine = x >= 1 && x <= P.nx - 2 && x >= P.ox0 - 1 && x <= P.ox0 + P.ow && !is_solid(P, x, y);
            if (!__any_sync(0xffffffffu, mine)) continue;
            if (mine) {
                T g[L::Q];
                unsigned links = 0u;
#pragma unroll
                for (int i = 0; i < L::Q; i++) {
                    g[i] = Store<S>::load(src, L::opp(i) * P.plane + row + x);
                    if (i > 0 && is_solid(P, x - L::cx(i), y - L::cy(i))) links |= 1u << i;
                }
                if (P.wall == WALL_DIFFUSE && links) diffuse_wall<L, T>(links, g);
#pragma unroll
                for (int i = 1; i < L::Q; i++)
                    if ((links >> i) & 1u) Store<S>::store(sb + i * LY::PLANE + c - L::cx(i), 0, g[i]);
            }
        }
    }
    // the stage is refilled by the async proxy after every warp has left it
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncwarp();
}

// u_x of the probe site of a staged row (the values the update read), logged
// for step t.  One lane calls.
template <typename S, int EQ, int R, int TX>
__device__ __noinline__ void log_probe(const Params& P, const S* box, int x0, long long t) {
    using L = D2Q9;
    using T = typename Store<S>::T;
    using LY = TmaLayout<S, R, TX>;
    const S* sb = box + (threadIdx.x >> 5) * LY::W + LY::H + (P.probe_x - x0);
    T g[L::Q], drho, rho, jx, jy, ux, uy;
#pragma unroll
    for (int i = 0; i < L::Q; i++) g[i] = Store<S>::load(sb + i * LY::PLANE - L::cx(i), 0);
    moments<L, T>(g, Par<T>::rho0(P), drho, rho, jx, jy);
    velocity<T>(jx, jy, rho, ux, uy);
    P.probe_ring[t % P.ring_cap] = (double)ux;
}

// One staged tile: rows y0 .. y0 + R - 1 and columns x0 .. x0 + TX - 1 of the
// run P, from box (the tile's staged source planes); warp w computes row
// y0 + w, lane l the site pairs x0 + 2 l + 64 s.  The updated sites go to sink.
// Pc: the parameters for the out-of-line paths (the same values as P, held
// where those paths read them fast).  state: what the warp carries on.
// Every row takes one path, the shifted shared-memory reads, after patch_row
// has put the boundary rules' populations into the rows that need any.  The
// sites that are not the tile's to update (the columns x = 0 and x = nx - 1,
// which edge_item updates, columns past the grid, the obstacle's sites) are
// updated from the rest state at unit density, whatever the staged planes
// hold, and are neither stored nor pending; solid sites hold zeros in both
// buffers from the start.
template <typename S, int EQ, int R, int TX = kTmaTX, typename Sink>
__device__ __forceinline__ void tma_tile(const Params& P, S* box, int x0, int y0, long long t,
                                         TileState<Sink>& state, MlpSlot<EQ>& mslot, const Params& Pc) {
    using L = D2Q9;
    using T = typename Store<S>::T;
    using LY = TmaLayout<S, R, TX>;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    S* __restrict__ dst = static_cast<S*>(P.dst);
    const int nxp = P.nxp, plane = (int)P.plane;
    const int y = y0 + warp;
    // one test clears almost every tile of the rows' own tests below
    const bool plain = !P.prestream && y0 >= 1 && y0 + R <= P.ny - 1 &&
                       (P.ow == 0 || x0 + TX < P.ox0 || x0 > P.ox0 + P.ow || y0 + R < P.oy0 || y0 > P.oy0 + P.oh);
    bool solid_row = false;
    if (!plain) {
        if (y >= P.ny) return;
        const bool near_obstacle = P.ow > 0 && y >= P.oy0 - 1 && y <= P.oy0 + P.oh && x0 + TX >= P.ox0 &&
                                   x0 <= P.ox0 + P.ow;
        if constexpr (sizeof(S) == 2) {
            if (near_obstacle && P.wall == WALL_DIFFUSE && !P.prestream) {
                state = tma_tile_general<S, EQ, R, TX>(Pc, box, x0, y0, t, state, mslot);
                return;
            }
        }
        if (P.prestream || y == 0 || y == P.ny - 1 || near_obstacle) patch_row<S, R, TX>(Pc, box, x0, y);
        solid_row = near_obstacle && y >= P.oy0 && y < P.oy0 + P.oh;
    }
    const S* sb = box + warp * LY::W + LY::H;
    const int row = y * nxp + x0;
    unsigned pmask = 0u;   // pending sites of the lane (bit 2 s + h: column 2 l + 64 s + h)
    const bool masked = x0 == 0 || x0 + TX >= P.nx || solid_row;   // uniform: some sites are not the row's
    // two adjacent sites per lane, columns c and c + 1 (c = 2 l + 64 s):
    // planes at rest and every store move both with one access, and the
    // two updates are one packed update, or (FP64) independent work for the
    // scheduler
#pragma unroll 1
    for (int s = 0; s < TX / 64; s++) {
        const int c = 2 * lane + 64 * s;
        bool ea = false, eb = false;   // not the row's sites
        if (masked) {
            const int x = x0 + c;
            ea = x == 0 || x >= P.nx - 1 || (solid_row && x >= P.ox0 && x < P.ox0 + P.ow);
            eb = x + 1 >= P.nx - 1 || (solid_row && x + 1 >= P.ox0 && x + 1 < P.ox0 + P.ow);
        }
        unsigned pend = 0u;
        T ga[L::Q], gb[L::Q];
#pragma unroll
        for (int i = 0; i < L::Q; i++) {
            const S* q = sb + i * LY::PLANE + c;
            if (L::cx(i) == 0) {
                PairIO<S>::load(q, ga[i], gb[i]);
            } else {
                ga[i] = Store<S>::load(q - L::cx(i), 0);
                gb[i] = Store<S>::load(q + 1 - L::cx(i), 0);
            }
        }
        if (masked) {
            const T r1 = T(1) - Par<T>::rho0(P);
#pragma unroll
            for (int i = 0; i < L::Q; i++) {
                ga[i] = ea ? T(L::w(i)) * r1 : ga[i];
                gb[i] = eb ? T(L::w(i)) * r1 : gb[i];
            }
        }
        // (the sites that are not the row's do not count as solved)
        float ma = 0.0f, mb = 0.0f;
        if constexpr (EQ == EQ_ENERGY_MLP) {
            ma = mlp_site_start<T>(P, mslot.s, true, ga);
            mb = mlp_site_start<T>(P, mslot.s, true, gb);
        }
        if constexpr (!kF64<T>) {
            f2 g[L::Q];
#pragma unroll
            for (int i = 0; i < L::Q; i++) g[i] = f2(ga[i], gb[i]);
            NewtonCount n2[2] = {};
            pend = update_pair<S, EQ>(P, g, state.nonfinite, n2, f2(ma, mb));
            if constexpr (EQ >= EQ_ENERGY) {
                if (!ea) state.nc.add(n2[0]);
                if (!eb) state.nc.add(n2[1]);
            }
#pragma unroll
            for (int i = 0; i < L::Q; i++) {
                ga[i] = g[i].x;
                gb[i] = g[i].y;
            }
        } else {
            NewtonCount na = state.nc;
            if (update_site<L, T, EQ, Store<S>::kProject, false>(P, ga, x0 + c, y, t, state.nonfinite, na, ma)) pend = 1u;
            if (EQ >= EQ_ENERGY && !ea) state.nc = na;
            na = state.nc;
            if (update_site<L, T, EQ, Store<S>::kProject, false>(P, gb, x0 + c + 1, y, t, state.nonfinite, na, mb))
                pend |= 2u;
            if (EQ >= EQ_ENERGY && !eb) state.nc = na;
        }
        if (!(ea | eb)) {
#pragma unroll
            for (int i = 0; i < L::Q; i++) {
                if constexpr (Store<S>::kPlain) {
                    const f2 w((float)L::w(i)), r = (f2(ga[i], gb[i]) + w) - w;   // store_round of both
                    PairIO<S>::store(dst + i * plane + row + c, r.x, r.y);
                } else {
                    PairIO<S>::store(dst + i * plane + row + c, ga[i], gb[i]);
                }
            }
        } else {
#pragma unroll
            for (int i = 0; i < L::Q; i++) {
                if (!ea) Store<S>::store(dst + i * plane + row + c, 0, store_round<L, S>(i, ga[i]));
                if (!eb) Store<S>::store(dst + i * plane + row + c + 1, 0, store_round<L, S>(i, gb[i]));
            }
        }
        pmask |= (pend & ((ea ? 0u : 1u) | (eb ? 0u : 2u))) << (2 * s);
    }
    // the row's pending sites, from the staged planes (valid until the warp
    // leaves the stage), out of line: the update keeps its registers
    if (__any_sync(0xffffffffu, pmask != 0u))
        state.sink = resolve_staged_row<S, EQ, R, TX>(Pc, box, x0, y, pmask, state.sink);
    if (P.probe_ring && y == P.probe_y && lane == 0 && P.probe_x >= x0 && P.probe_x < x0 + TX &&
        P.probe_x >= 1 && P.probe_x <= P.nx - 2 && !is_solid(P, P.probe_x, y))
        log_probe<S, EQ, R, TX>(Pc, box, x0, t);
}
// Resident blocks per SM the staged kernel is compiled for: two in general
// (128 registers per thread with 8-row tiles, 170 with 6-row tiles); three
// (85 registers per thread) for FP32 tiles 64 sites wide, which take half the
// shared memory.
template <typename S, int EQ, int R, int TX>
constexpr int tma_min_blocks() {
    if (EQ >= EQ_ENERGY) return 2;   // (the packed solve spills at 85)
    return sizeof(S) == 4 && TX == 64 && R == 8 ? 3 : 2;
}

// Stages of the 8-row tiles: two fill the shared memory two blocks share; FP16
// storage has room for a third (us per step of two runs side by side, 4096 x
// 2048, polynomial f*: 65.6; two stages and three blocks, 85 registers: 69.0;
// four stages: 67.1; entropic f*: 86.0; 130.6; 91.3).
template <typename S>
constexpr int kStages8 = sizeof(S) == 2 ? 3 : 2;

template <typename S, int EQ, int R, int STAGES, int TX = kTmaTX>
__global__ void __launch_bounds__(32 * R, tma_min_blocks<S, EQ, R, TX>())
    k_collide_d2q9_tma(const __grid_constant__ Params P, const __grid_constant__ CUtensorMap tm) {
    using L = D2Q9;
    using T = typename Store<S>::T;
    using LY = TmaLayout<S, R, TX>;
    extern __shared__ unsigned char smem_raw[];
    unsigned char* smem = smem_raw + ((128 - (smem_u32(smem_raw) & 127)) & 127);
    S* stages = reinterpret_cast<S*>(smem);
    unsigned long long* full = reinterpret_cast<unsigned long long*>(smem + STAGES * LY::STAGE_BYTES);
    unsigned long long* gather = full + STAGES;   // the warps' rendezvous before a cut
    constexpr int kCap = tma_cand_cap<R, TX>();
    constexpr int kRoom = kCap - TX * R;
    using Shared = TmaShared<kCap>;
    Shared& sh = *reinterpret_cast<Shared*>(smem + STAGES * LY::STAGE_BYTES + 8 * (STAGES + 1));
    constexpr size_t kMlpOff = (STAGES * LY::STAGE_BYTES + 8 * (STAGES + 1) + sizeof(Shared) + 15) / 16 * 16;
    MlpSlot<EQ>& mslot = *reinterpret_cast<MlpSlot<EQ>*>(smem + kMlpOff);
    if (threadIdx.x == 0) {
        for (int st = 0; st < STAGES; st++) {
            mbar_init(&full[st], 1);
            sh.ring.done[st] = 0;
        }
        mbar_init(gather, R);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        sh.p = P;
        sh.abort = 0;
        sh.begun = 0u;
        sh.met = 0u;
        sh.bc.n = 0;
    }
    const int tiles_x = (P.nx + TX - 1) / TX;
    const int tiles = tiles_x * ((P.ny + R - 1) / R);
    // the x = 0 and x = nx - 1 columns go first, as edge items of 32 R sites
    const int edge_items = ((P.nx > 1 ? 2 : 1) * P.ny + 32 * R - 1) / (32 * R);

    // Work is handed out by claims: claim c < edge_items is edge item c, the
    // others tile tile_order[c - edge_items] (the tiles with rows to patch
    // first) or c - edge_items.  A block's first STAGES claims are fixed
    // (b, b + G, b + 2 G, ... for block b of G): the pipeline fills without
    // waiting for the atomic; the counter hands out the claims from STAGES G
    // on.  Thread 0 claims two refills ahead and reads the claim's order
    // entry one ahead (both latencies then overlap a tile's computation), and
    // publishes it before it leaves the stage it will refill.
    int claimed = 0;   // thread 0: a claim
    int next = 0;      // thread 0: the claim before it, as work: a tile, -2 - e for edge item e, -1 for none
    auto resolve = [&]() {
        const int c = claimed - edge_items;
        next = c < 0 ? -2 - claimed : c < tiles ? c : -1;
        if (P.tile_order && c >= 0 && c < tiles) next = __ldg(P.tile_order + c);
    };
    if (threadIdx.x == 0) {
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<unsigned long long>(&tm)) : "memory");
        for (int st = 0; st < STAGES; st++) {
            claimed = (int)blockIdx.x + st * (int)gridDim.x;
            resolve();
            sh.ring.next[st] = next;
        }
    }
    // Launched as a programmatic dependent of the previous kernel in the
    // stream: the block may start while that kernel finishes, and the code
    // above reads only the launch's parameters and the claim order (which no
    // kernel writes) and writes only shared memory.  Every thread waits here
    // until the previous kernel has completed and its writes are visible.
    // (The next kernel's blocks are let in when this one's have finished their
    // tiles, to wait here in turn: let in at the start, they only take room
    // from other streams' kernels.)
    asm volatile("griddepcontrol.wait;" ::: "memory");
    mslot.fill(P);
    __syncthreads();
    const long long t = *P.step;

    auto claim = [&]() { claimed = (int)atomicAdd(P.tile_counter, 1u) + STAGES * (int)gridDim.x; };
    // One thread: put the claimed work into a stage (the phase of an edge
    // item, or of no work, is completed by a plain arrive, without a copy).
    auto fill = [&](int st) {
        unsigned long long* bar = &full[st];
        const int tile = sh.ring.next[st];
        sh.ring.tile[st] = tile;
        if (tile < 0) {
            asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
            return;
        }
        const int ty = tile / tiles_x, tx = tile - ty * tiles_x;
        sh.ring.x0[st] = tx * TX;
        sh.ring.y0[st] = ty * R;
        mbar_expect_tx(bar, (unsigned)LY::TX_BYTES);
        S* base = stages + (size_t)st * (LY::STAGE_BYTES / sizeof(S));
#pragma unroll
        for (int i = 0; i < L::Q; i++)
            tma_load_3d(base + i * LY::PLANE, &tm, tx * TX - LY::H, ty * R - L::cy(i), i, bar);
    };
    if (threadIdx.x == 0) {
        for (int st = 0; st < STAGES; st++) fill(st);
        claim();
        resolve();
        claim();
    }
    // The sites the dS bound does not clear are resolved as they are
    // updated; the candidates go to the block's buffer.  A warp that finds it
    // filling up asks for a cut: before the first work that no warp has begun
    // by then, the warps meet and cut the buffer to its k best (or flush it,
    // where k does not fit).  The warps are at most STAGES tiles apart; what
    // a tile begun before the cut finds no room for goes to the global list.
    const int kept = P.k > 0 && P.k < kRoom ? P.k : 0;
    const unsigned cut_above = (unsigned)(kept + (kRoom - kept) / 2);
    TileState<CandSink<kCap>> state{{&sh.bc}, {0, 0, 0, 0}, false};
    int st = 0;
    unsigned parity = 0u, cuts = 0u;
    for (unsigned jj = 1u;; jj++) {
        // one atomic both announces the work as begun and finds a cut asked
        // for before it (the asking bit outranks every ordinal, and freezes
        // the one it found), so every warp cuts before the same work; its
        // latency passes with the wait
        unsigned begun = 0u;
        if ((threadIdx.x & 31) == 0) begun = atomicMax(&sh.begun, jj);
        // a warp whose wait gives up (here or below) leaves its stage held, so
        // that every other warp's wait gives up in turn; the one reduction
        // hands lane 0's finding to the warp and makes a lane's expired wait
        // the warp's (kGaveUp outranks every finding)
        if (!mbar_wait(&full[st], parity)) begun = kGaveUp;
        begun = __reduce_max_sync(0xffffffffu, begun);
        if (begun == kGaveUp) {
            sh.abort = 1;
            break;
        }
        const int tile = sh.ring.tile[st];
        if (tile == -1) break;
        if (threadIdx.x == 0) {
            sh.ring.next[st] = next;
            resolve();
            claim();
        }
        if (begun >= kCutAsked && jj > (begun & ~kCutAsked)) {
            if ((threadIdx.x & 31) == 0)
                asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(gather)) : "memory");
            // one outcome for the block, also where some warps' waits gave up
            // and the others' did not: the cut's barriers need every warp
            const bool met = warp_wait(gather, cuts & 1u);
            bool cut = false;
            if ((threadIdx.x & 31) == 0)
                cut = rendezvous_met(met, cuts, [&](unsigned e, unsigned d) { return atomicCAS(&sh.met, e, d); });
            if (!__shfl_sync(0xffffffffu, (int)cut, 0)) {
                sh.abort = 1;
                break;
            }
            cuts++;
            if (P.k < kRoom) block_cut(sh.bc, sh.ss.sc, P.k);
            else block_flush(sh.p, sh.bc);
            if (threadIdx.x == 0) sh.begun = jj;
            __syncthreads();
        }
        if (tile <= -2) {
            state = edge_item<S, EQ, R>(sh.p, -2 - tile, t, state, mslot);
        } else {
            S* box = stages + (size_t)st * (LY::STAGE_BYTES / sizeof(S));
            tma_tile<S, EQ, R, TX>(P, box, sh.ring.x0[st], sh.ring.y0[st], t, state, mslot, sh.p);
        }
        __syncwarp();
        if ((threadIdx.x & 31) == 0) {
            if (sh.bc.n > cut_above) atomicOr(&sh.begun, kCutAsked);
            if (stage_leave(&sh.ring.done[st], R)) fill(st);
        }
        if (++st == STAGES) {
            st = 0;
            parity ^= 1u;
        }
    }
    __syncthreads();
    if (sh.abort && threadIdx.x == 0) {
        atomicOr(P.err, ERR_TIMEOUT);
        // wait (bounded) for copies still in flight into every stage
        for (int k2 = 0; k2 < STAGES; k2++) {
            mbar_wait(&full[st], parity);
            if (++st == STAGES) {
                st = 0;
                parity ^= 1u;
            }
        }
    }
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (state.nonfinite) atomicOr(P.err, ERR_NONFINITE);
    if constexpr (EQ >= EQ_ENERGY) flush_newton(P, state.nc);
    // the staged tiles are no longer needed: their memory holds the last
    // block's candidate staging
    const int scap = (int)min((size_t)kStage, (size_t)STAGES * LY::STAGE_BYTES / 12);
    unsigned long long* skey = reinterpret_cast<unsigned long long*>(smem);
    unsigned* sidx = reinterpret_cast<unsigned*>(smem + 8 * scap);
    finish_parts<L, S, EQ>(sh.p, sh.is_last, sh.ss, sh.bc, skey, sidx, scap);
}

// ---------------------------------------------------------------------------
// K1, one site per thread (D1Q3).
// ---------------------------------------------------------------------------
template <typename L, typename S, int EQ>
__global__ void __launch_bounds__(kSiteBlock) k_collide_site(const __grid_constant__ Params P) {
    using T = typename Store<S>::T;
    __shared__ SiteShared<kBlockCand> sh;   // room for the block's sites
    static_assert(kBlockCand >= kSiteBlock, "every site of the block may be a candidate");
    if (threadIdx.x == 0) {
        sh.p = P;
        sh.bc.n = 0;
    }
    __syncthreads();
    const long long t = *P.step;
    const long long sid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const int x = (int)(sid % P.nx), y = (int)(sid / P.nx);
    const bool inside = sid < (long long)P.nx * P.ny;
    const bool valid = inside && !is_solid(P, x, y);
    bool nonfinite = false, pending = false;
    NewtonCount nc = {0, 0, 0, 0};
    T g[L::Q];
    if (valid) {
        gather_site<L, S>(P, x, y, g);
        pending = update_site<L, T, EQ, Store<S>::kProject>(P, g, x, y, t, nonfinite, nc);
    }
    if (inside) {
        const long long o = (long long)y * P.nxp + x;
#pragma unroll
        for (int i = 0; i < L::Q; i++)
            Store<S>::store(P.dst, i * P.plane + o, valid ? store_round<L, S>(i, g[i]) : T(0));
    }
    if (__any_sync(0xffffffffu, pending)) {
        T ds = T(-1);
        if (pending) ds = resolve_ds<L, S, EQ>(sh.p, x, y);
        block_push<T>(P, sh.bc, ds > Par<T>::delta(P), ds, (unsigned)sid);
    }
    if (nonfinite) atomicOr(P.err, ERR_NONFINITE);
    finish_parts<L, S, EQ>(sh.p, sh.is_last, sh.ss, sh.bc, sh.key, sh.idx, kStage);
}

// ---------------------------------------------------------------------------
// K1 for short D1Q3 runs: many time steps in one launch of one cluster.
// A few hundred sites leave no work to spread: what bounds a step is its
// chain -- launch, loads, the FP64 update (two FP64 operations per SM and
// clock), the exact dS of the sites near the front, the selection -- so the
// state stays in the shared memory of a cluster of 16 blocks (16 SMs' FP64
// pipes), neighbours read each other's edge sites there, every block lists its
// candidates and gives them their f* at once, and the hardware's cluster
// barrier separates the collision from the selection; only a step with more
// than k candidates, where some take their post-collision populations back,
// needs a second one before the next free flight.  The exact dS of a warp's
// pending sites takes a lane per population (its series are the longest FP64
// chain of a step).
// 800 sites, FP64: 19.5 us per step in one launch each (13 blocks), 6.1 us so
// (2.5 us without the selection).
// Every population passes through the storage type, so results are those of
// one launch per step.
// ---------------------------------------------------------------------------
constexpr int kTubeBlocks = 16;          // cluster size
constexpr int kTubeThreads = 256;        // most sites per block
constexpr int kTubeRank = 128;           // candidates ranked by counting

template <typename T>
struct TubeShared {
    TopkScratch sc;
    Thresh th;
    unsigned count[3];                   // the block's candidates of step t in count[t mod 3]
    unsigned long long key[kTubeThreads];
    unsigned idx[kTubeThreads];
    T pend[kTubeThreads / 32][32][6];    // per warp: g and f* of its pending sites, then dS
};

template <typename S>
constexpr size_t tube_smem_bytes(int n) {
    const int per = (n + kTubeBlocks - 1) / kTubeBlocks;
    return (size_t)n * 12 + 16 + 6 * (size_t)per * sizeof(S);
}

// Exact dS (delta_s_exact, the same operations) of the warp's pending sites,
// a lane per population: slot[j] holds g and f* of the warp's j-th pending
// site.  Every lane calls; returns the lane's dS (-1: not pending).
template <typename T>
__device__ __forceinline__ T warp_delta_s(bool pending, const T* g, const T* gs, T rho0, T (*slot)[6]) {
    using L = D1Q3;
    const int lane = threadIdx.x & 31;
    const unsigned mask = __ballot_sync(0xffffffffu, pending);
    const int n = __popc(mask), own = __popc(mask & ((1u << lane) - 1u));
    if (pending)
#pragma unroll
        for (int i = 0; i < L::Q; i++) {
            slot[own][i] = g[i];
            slot[own][3 + i] = gs[i];
        }
    __syncwarp();
    const int part = lane % 3;
    const T w = part == 0 ? T(L::w(0)) : T(L::w(1));
    for (int b = 0; b < n; b += 10) {
        const int j = b + lane / 3;
        const bool on = lane < 30 && j < n;
        T fs = T(1), x = T(0);
        bool bad = false;
        if (on) {
            const T gi = slot[j][part], si = slot[j][3 + part];
            fs = dfma<T>(w, rho0, si);
            const T f = dfma<T>(w, rho0, gi);
            bad = !(fs > T(0)) || (f < T(0));
            if constexpr (kF64<T>) x = (gi - si) * recip<T>(fs);
            else x = (gi - si) / fs;
        }
        const T phi = bad ? T(0) : phi_fn<T>(x);
        const T fs1 = __shfl_down_sync(0xffffffffu, fs, 1), fs2 = __shfl_down_sync(0xffffffffu, fs, 2);
        const T phi1 = __shfl_down_sync(0xffffffffu, phi, 1), phi2 = __shfl_down_sync(0xffffffffu, phi, 2);
        const unsigned bads = __ballot_sync(0xffffffffu, bad);
        if (on && part == 0) {
            const T ds = dfma<T>(fs2, phi2, dfma<T>(fs1, phi1, dfma<T>(fs, phi, T(0))));
            slot[j][0] = (bads >> lane) & 7u ? T(INFINITY) : ds;
        }
        __syncwarp();
    }
    return pending ? slot[own][0] : T(-1);
}

__device__ __forceinline__ void cluster_arrive() {
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
    __syncwarp();
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

template <typename S, int EQ>
__global__ void __launch_bounds__(kTubeThreads) k_tube(const __grid_constant__ Params P, int steps, void* out) {
    using L = D1Q3;
    using T = typename Store<S>::T;
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    extern __shared__ __align__(16) unsigned char tube_raw[];
    __shared__ TubeShared<T> sh;
    const int n = P.nx, per = (n + kTubeBlocks - 1) / kTubeBlocks;
    const int rank = (int)cluster.block_rank(), tid = threadIdx.x, lane = tid & 31;
    const int x = rank * per + tid;
    const bool mine = tid < per && x < n;
    // block 0: a step's candidates when they are ranked by radix; every block:
    // its sites' post-collision populations [parity][plane][per]
    unsigned long long* key = reinterpret_cast<unsigned long long*>(tube_raw);
    unsigned* idx = reinterpret_cast<unsigned*>(tube_raw + (size_t)n * 8);
    S* f = reinterpret_cast<S*>(tube_raw + ((size_t)n * 12 + 15) / 16 * 16);
    if (tid < 3) sh.count[tid] = 0u;
    if (mine)
#pragma unroll
        for (int i = 0; i < L::Q; i++) f[i * per + tid] = static_cast<const S*>(P.src)[i * P.plane + x];
    const long long t0 = *P.step;
    const T delta = Par<T>::delta(P), rho0 = Par<T>::rho0(P);
    bool nonfinite = false;
    NewtonCount nc = {0, 0, 0, 0};
    int c = (int)(t0 % 3), ring = (int)(t0 % P.ring_cap);
    cluster.sync();
    for (int s = 0; s < steps; s++) {
        S* cur = f + (s & 1) * 3 * per;
        S* nxt = f + ((s + 1) & 1) * 3 * per;
        // population i of site xx after the previous step
        auto at = [&](int i, int xx) {
            const int b = xx / per;
            const S* q = b == rank ? cur : cluster.map_shared_rank(cur, b);
            return Store<S>::load(q + i * per + xx - b * per, 0);
        };
        bool pending = false;
        T g[L::Q], pre[L::Q], gs[L::Q];
        if (mine) {
            if (s == 0 && P.prestream) {
#pragma unroll
                for (int i = 0; i < L::Q; i++) g[i] = at(i, x);
            } else {
                // free flight with the rules of gather_site
                g[0] = at(0, x);
#pragma unroll
                for (int i = 1; i < L::Q; i++) {
                    const int sx = x - L::cx(i), local = tid - L::cx(i);
                    if (local >= 0 && local < per && sx < n) {
                        g[i] = Store<S>::load(cur + i * per + local, 0);
                        continue;
                    }
                    if (sx >= 0 && sx < n) {
                        g[i] = at(i, sx);
                        continue;
                    }
                    const int kind = sx < 0 ? P.bc[0] : P.bc[1];
                    if (kind == BC_PERIODIC) {
                        g[i] = at(i, sx < 0 ? sx + n : sx - n);
                    } else if (kind == BC_INLET) {
                        g[i] = (T)P.gin[i];
                    } else if (kind == BC_OUTLET) {
                        T v[L::Q], go[L::Q];
#pragma unroll
                        for (int j = 0; j < L::Q; j++) v[j] = at(j, n - 2);
                        outlet_equilibrium<L, T>(P, v, go);
                        g[i] = store_round<L, S>(i, go[i]);
                    } else if (kind == BC_OUTLET_COPY) {
                        g[i] = at(i, x);
                    } else {
                        g[i] = at(L::opp(i), x);
                    }
                }
            }
#pragma unroll
            for (int i = 0; i < L::Q; i++) pre[i] = g[i];
            pending = update_site<L, T, EQ, Store<S>::kProject>(P, g, x, 0, t0 + s, nonfinite, nc, 0.0f, nullptr, gs);
#pragma unroll
            for (int i = 0; i < L::Q; i++) Store<S>::store(nxt + i * per + tid, 0, store_round<L, S>(i, g[i]));
        }
        T ds = T(-1);
        if (__any_sync(0xffffffffu, pending)) {
            ds = warp_delta_s<T>(pending, pre, gs, rho0, sh.pend[tid >> 5]);
            if (pending) {
                PopArr<L::Q, T> pa;
#pragma unroll
                for (int i = 0; i < L::Q; i++) pa.v[i] = pre[i];
                ds = recheck_ds<L, T, EQ>(pa, ds, delta, P.delta, P.rho0, P.recheck_band, P.recheck);
            }
        }
        const bool cand = ds > delta;
        const unsigned long long k = cand ? ds_key((double)ds) : 0ull;
        unsigned slot = 0u;
        if (cand) {
            slot = atomicAdd(sh.count + c, 1u);
            sh.key[slot] = k;
            sh.idx[slot] = (unsigned)x;
        }
        // the next step's counter: last read two steps ago, before the
        // previous step's barrier
        const int cn = c == 2 ? 0 : c + 1;
        if (tid == 0) sh.count[cn] = 0u;
        if (cand) {
            // the Ehrenfests' step from the stored post-collision populations,
            // as if every candidate were selected; with more than k of them
            // the others take theirs (g) back
            T h[L::Q];
#pragma unroll
            for (int i = 0; i < L::Q; i++) h[i] = Store<S>::load(nxt + i * per + tid, 0);
            ehrenfest_value<L, S, EQ>(P, h);
#pragma unroll
            for (int i = 0; i < L::Q; i++) Store<S>::store(nxt + i * per + tid, 0, store_round<L, S>(i, h[i]));
        }
        cluster_arrive();
        cluster_wait();
        // every block's count, in lanes 0 .. 15; m: the step's candidates
        // (the same for every thread)
        int m = 0;
        unsigned cnt = 0u;
        if (P.k > 0) {
            if (lane < kTubeBlocks) cnt = cluster.map_shared_rank(sh.count, lane)[c];
            m = (int)__reduce_add_sync(0xffffffffu, cnt);
        }
        if (m > 0) {
            bool take = cand;
            if (m <= P.k) {
                slot += __reduce_add_sync(0xffffffffu, lane < rank ? cnt : 0u);
            } else if (m <= kTubeRank) {
                if (__any_sync(0xffffffffu, cand)) {
                    slot = 0u;
                    for (int b = 0; b < kTubeBlocks; b++) {
                        const int nb = (int)__shfl_sync(0xffffffffu, cnt, b);
                        const unsigned long long* kb = cluster.map_shared_rank(sh.key, b);
                        const unsigned* ib = cluster.map_shared_rank(sh.idx, b);
                        for (int e = 0; e < nb; e++) {
                            const unsigned long long ke = kb[e];
                            slot += ke > k || (ke == k && ib[e] < (unsigned)x);
                        }
                    }
                    take = cand && slot < (unsigned)P.k;
                }
            } else {
                if (rank == 0) {
                    int base = 0;
                    for (int b = 0; b < kTubeBlocks; b++) {
                        const int nb = (int)__shfl_sync(0xffffffffu, cnt, b);
                        const unsigned long long* kb = cluster.map_shared_rank(sh.key, b);
                        const unsigned* ib = cluster.map_shared_rank(sh.idx, b);
                        for (int e = tid; e < nb; e += blockDim.x) {
                            key[base + e] = kb[e];
                            idx[base + e] = ib[e];
                        }
                        base += nb;
                    }
                    __syncthreads();
                    const Thresh th = block_topk(sh.sc, m, P.k, [&](int e) { return key[e]; },
                                                 [&](int e) { return idx[e]; });
                    if (tid == 0) sh.th = th;
                }
                cluster.sync();
                const Thresh th = *cluster.map_shared_rank(&sh.th, 0);
                take = cand && th.selected(k, (unsigned)x);
                if (take && s == steps - 1) {
                    // its place in the list: its rank among the selected
                    const unsigned long long* key0 = cluster.map_shared_rank(key, 0);
                    const unsigned* idx0 = cluster.map_shared_rank(idx, 0);
                    slot = 0u;
                    for (int e = 0; e < m; e++) slot += idx0[e] < (unsigned)x && th.selected(key0[e], idx0[e]);
                }
            }
            if (take && s == steps - 1) P.sel_idx[slot] = x;   // (order unspecified)
            if (m > P.k) {
                if (cand && !take)
#pragma unroll
                    for (int i = 0; i < L::Q; i++)
                        Store<S>::store(nxt + i * per + tid, 0, store_round<L, S>(i, g[i]));
                cluster_arrive();
                cluster_wait();
            }
        }
        if (rank == 0 && tid == 0) {
            P.count_ring[ring] = min(m, P.k);
            if (s == steps - 1) {
                *P.sel_count = min(m, P.k);
                *P.step = t0 + steps;
            }
        }
        c = cn;
        ring = ring + 1 == P.ring_cap ? 0 : ring + 1;
    }
    if (mine) {
        const S* last = f + (steps & 1) * 3 * per;
#pragma unroll
        for (int i = 0; i < L::Q; i++) static_cast<S*>(out)[i * P.plane + x] = last[i * per + tid];
    }
    if (nonfinite) atomicOr(P.err, ERR_NONFINITE);
    // no block leaves while another may still read its shared memory
    cluster.sync();
}

// Stand-alone selection (select-only test hook).
template <typename L, typename S, int EQ>
__global__ void __launch_bounds__(kSelectThreads) k_select(const __grid_constant__ Params P, int stage_cap,
                                                           int mode) {
    extern __shared__ unsigned long long dyn[];
    __shared__ SelectShared ss;
    select_and_fix<L, S, EQ>(P, ss, dyn, reinterpret_cast<unsigned*>(dyn + stage_cap), stage_cap, mode);
}

#ifdef LBM_DEFINE_EMIT_FROM_DS
// Candidates from a given dS array (select-only test hook): each block of
// 256 threads takes kEmitPerBlock consecutive values through the same block
// stage as K1 (its k best reach the global list).
constexpr int kEmitPerBlock = 2048;
__global__ void __launch_bounds__(256) k_emit_from_ds(const __grid_constant__ Params P, const double* ds,
                                                      int n) {
    __shared__ BlockCand bc;
    __shared__ TopkScratch sc;
    if (threadIdx.x == 0) bc.n = 0;
    if (P.k <= 0) return;
    const long long b0 = (long long)blockIdx.x * kEmitPerBlock;
    for (int r = 0; r < kEmitPerBlock; r += 256) {
        block_room(P, bc, sc);
        const long long i = b0 + r + threadIdx.x;
        const double v = i < n ? ds[i] : -INFINITY;
        block_push<double>(P, bc, i < n && v > P.delta, v, (unsigned)i);
    }
    block_finish(P, bc, sc);
}
#endif

// ---------------------------------------------------------------------------
// State import / export and field kernels (one site per thread).
// ---------------------------------------------------------------------------

// Quasiequilibrium of given (rho, u) at every fluid site; zero elsewhere.
template <typename L, typename S, int EQ>
__global__ void k_init_eq(const __grid_constant__ Params P, const double* rho, const double* ux,
                          const double* uy, const double* e2) {
    using T = typename Store<S>::T;
    const long long sid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (sid >= (long long)P.nx * P.ny) return;
    const int y = (int)((unsigned)sid / (unsigned)P.nx), x = (int)((unsigned)sid - (unsigned)y * P.nx);   // (< 2^31 sites)
    const long long o = (long long)y * P.nxp + x;
    T gs[L::Q];
    if (is_solid(P, x, y)) {
#pragma unroll
        for (int i = 0; i < L::Q; i++) gs[i] = T(0);
    } else {
        const double v = uy ? uy[sid] : 0.0;
        bool done = false;
        if constexpr (EQ >= EQ_ENERGY) {
            if (e2) {
                const T r = T(rho[sid]), u = T(ux[sid]);
                NewtonCount nc = {0, 0, 0, 0};
                equilibrium_energy<T, EQ>(r, r * u, r * T(v), T(e2[sid]), gs, nc);
#pragma unroll
                for (int i = 0; i < L::Q; i++) gs[i] = store_round<L, S>(i, gs[i]);
                done = true;
            }
        }
        // polynomial or entropic f* (the energy forms without a given energy:
        // the isothermal entropic formula) in FP64, held as the storage
        // holds it
        if (!done) bc_equilibrium<L, S>(P, rho[sid], ux[sid], v, gs);
    }
#pragma unroll
    for (int i = 0; i < L::Q; i++) Store<S>::store(P.dst, i * P.plane + o, gs[i]);
}

// FP64 populations [Q][ny][nx] -> deviation storage, planes [i0, i1).
template <typename L, typename S>
__global__ void k_import(const __grid_constant__ Params P, const double* f, int i0, int i1) {
    const long long N = (long long)P.nx * P.ny;
    const long long sid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (sid >= N) return;
    const int y = (int)((unsigned)sid / (unsigned)P.nx), x = (int)((unsigned)sid - (unsigned)y * P.nx);   // (< 2^31 sites)
    const long long o = (long long)y * P.nxp + x;
    const bool solid = is_solid(P, x, y);
    using T = typename Store<S>::T;
    if (P.rho0 == 0.0) {
        // FP64 storage: a copy (no FP64 arithmetic)
#pragma unroll
        for (int i = 0; i < L::Q; i++)
            if (i >= i0 && i < i1) Store<S>::store(P.dst, i * P.plane + o, (T)(solid ? 0.0 : f[i * N + sid]));
        return;
    }
#pragma unroll
    for (int i = 0; i < L::Q; i++)
        if (i >= i0 && i < i1)
            Store<S>::store(P.dst, i * P.plane + o, solid ? T(0) : dev_of_f64<L, S>(P, i, f[i * N + sid]));
}

// Running sum s + c of floats: s their rounded sum, c the sum of the
// rounding errors (two-sum).
struct Sum2 {
    float s, c;
    __device__ __forceinline__ void add(float x) {
        const ff t = ff_two_sum(s, x);
        s = t.hi;
        c += t.lo;
    }
    __device__ __forceinline__ void add(Sum2 o) {
        add(o.s);
        c += o.c;
    }
    __device__ __forceinline__ ff value() const { return ff_fast_two_sum(s, c); }
};

// Pre-collision state of the current step (gather of src) at sites
// [s0, s1), exported as mode 0: populations f [Q][ny][nx]; 1: rho, ux, uy,
// 2E; 2: exact dS (outputs indexed by the site's index y nx + x).
// The moments of FP32 / FP16 storage were bound by the FP64 pipe (27
// operations per site, conversions included); six are left, the sums share
// their parts, and the conversions run on the integer pipe (a predicated
// conversion instruction still took its FP64 slots): 4096 x 2048, FP32:
// 355 -> 222 -> 144 us, FP64 2048 x 1024 (divisions and products with lattice
// velocities before): 302 -> 100 us.
template <typename L, typename S, int EQ>
__global__ void k_export(const __grid_constant__ Params P, int mode, double* o0, double* o1, double* o2,
                         double* o3, long long s0, long long s1) {
    using T = typename Store<S>::T;
    const long long N = (long long)P.nx * P.ny;
    const long long sid = s0 + (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (sid >= s1) return;
    const int y = (int)((unsigned)sid / (unsigned)P.nx), x = (int)((unsigned)sid - (unsigned)y * P.nx);   // (< 2^31 sites)
    if (is_solid(P, x, y)) {
        if (mode == 0) for (int i = 0; i < L::Q; i++) o0[i * N + sid] = 0.0;
        if (mode == 1) {
            o0[sid] = 0.0;
            if (o1) o1[sid] = 0.0;
            if (o2) o2[sid] = 0.0;
            if (o3) o3[sid] = 0.0;
        }
        if (mode == 2) o0[sid] = __longlong_as_double(0x7ff8000000000000ll);
        return;
    }
    T g[L::Q];
    gather_site<L, S>(P, x, y, g);
    if (mode == 0) {
#pragma unroll
        for (int i = 0; i < L::Q; i++) o0[i * N + sid] = pop_f64<L, S>(i, g[i]);
    } else if (mode == 1) {
        if constexpr (sizeof(T) == 4) {
            // FP32 / FP16 storage: the sums of the stored values in float-float
            // and u = j / rho by one corrected FP32 quotient, so that FP64
            // sees one addition per part; the rho0 parts (sum W = 1,
            // sum W v = 0, sum W |v|^2) are added in FP64 at the end.
            Sum2 one = {0.0f, 0.0f}, two = {0.0f, 0.0f}, jxs = {0.0f, 0.0f}, jys = {0.0f, 0.0f};
            bool first1 = true, first2 = true, firstx = true, firsty = true;
#pragma unroll
            for (int i = 1; i < L::Q; i++) {
                const int c2 = L::cx(i) * L::cx(i) + L::cy(i) * L::cy(i);
                auto put = [](Sum2& a, bool& first, float v) {
                    if (first) a.s = v;
                    else a.add(v);
                    first = false;
                };
                if (c2 == 1) put(one, first1, g[i]);
                if (c2 == 2) put(two, first2, g[i]);
                if (L::cx(i) != 0) put(jxs, firstx, L::cx(i) > 0 ? g[i] : -g[i]);
                if (L::cy(i) != 0) put(jys, firsty, L::cy(i) > 0 ? g[i] : -g[i]);
            }
            Sum2 rs = {g[0], 0.0f}, es = one;
            rs.add(one);
            if constexpr (L::Q == 9) {
                rs.add(two);
                es.add(Sum2{2.0f * two.s, 2.0f * two.c});
            }
            const ff r = rs.value(), jx = jxs.value(), jy = jys.value(), e = es.value();
            // the stored deviations' offsets: sum W rho0 (= rho0), and for
            // plain FP32 the sums of the FP32 weights (exact in FP64)
            constexpr bool plain = Store<S>::kPlain;
            constexpr float w0 = (float)L::w(0), w1 = (float)L::w(1), w5 = L::Q == 9 ? (float)L::w(L::Q - 1) : 0.0f;
            constexpr int n1 = L::Q == 9 ? 4 : 2, n2 = L::Q == 9 ? 4 : 0;
            constexpr double off0 = plain ? (double)w0 + n1 * (double)w1 + n2 * (double)w5 : 1.0;
            constexpr double off2 = plain ? n1 * (double)w1 + 2 * n2 * (double)w5 : L::sum_w_c2;
            constexpr float off0h = (float)off0, off0l = (float)(off0 - (double)off0h);
            o0[sid] = (off0 + widen(r.hi)) + widen(r.lo);
            const ff ir = ff_recip(ff_add({off0h, off0l}, r));
            if (o1) {
                const ff u = ff_mul(jx, ir);
                o1[sid] = widen(u.hi) + widen(u.lo);
            }
            if (o2) {
                const ff v = ff_mul(jy, ir);
                o2[sid] = widen(v.hi) + widen(v.lo);
            }
            if (o3) o3[sid] = (off2 + widen(e.hi)) + widen(e.lo);
        } else {
            double drho, rho, jx, jy, ux, uy;
            moments<L, double>(g, 0.0, drho, rho, jx, jy);
            velocity<double>(jx, jy, drho, ux, uy);
            o0[sid] = drho;
            if (o1) o1[sid] = ux;
            if (o2) o2[sid] = uy;
            if (o3) {
                if constexpr (L::Q == 9)
                    o3[sid] = fma(2.0, (g[5] + g[8]) + (g[6] + g[7]), (g[1] + g[3]) + (g[2] + g[4]));
                else
                    o3[sid] = g[1] + g[2];
            }
        }
    } else {
        T gs[L::Q], rho, ux, uy;
        site_equilibrium<L, T, EQ>(P, g, gs, rho, ux, uy);
        o0[sid] = (double)delta_s_exact<L, T>(g, gs, Par<T>::rho0(P));
    }
}

// Ghost exchange of a slab (runs sharded in x): copies the three
// populations that cross a face -- moving right (v_x = +1: 1, 5, 8) or left
// (v_x = -1: 3, 6, 7) -- of column col of the field, between the field and
// a packed buffer [3][ny] (dir 0: field -> buffer; 1: buffer -> field).
template <typename S>
__global__ void k_ghost(const __grid_constant__ Params P, S* field, int col, int right, S* buf, int dir) {
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= 3 * P.ny) return;
    const int p = j / P.ny, y = j - p * P.ny;
    const int plane = right ? (p == 0 ? 1 : (p == 1 ? 5 : 8)) : (p == 0 ? 3 : (p == 1 ? 6 : 7));
    S* at = field + plane * P.plane + (long long)y * P.nxp + col;
    if (dir == 0) buf[j] = *at;
    else *at = buf[j];
}

// ---------------------------------------------------------------------------
// Launchers for one storage type.  Tile shapes of the D2Q9 kernel (sites per
// thread in x, warps per block, minimum resident blocks per SM):
//   0: 1, 8, 3     1: 1, 8, 4     2: 2, 8, 2     3: 4, 8, 1
// and of the staged kernel (rows x columns per block tile, tiles in flight):
//   4: 8 x 128, 2 (FP16: 3)     5: 6 x 128, 3     6: 8 x 64, 2
// The persistent grid is (resident blocks per SM) x (SM count), from the
// occupancy calculator, capped by the number of tiles (small grids then
// spread over as many SMs as they have tiles: their step is latency-bound).
// ---------------------------------------------------------------------------
// Launch with programmatic stream serialisation: it may begin before the
// previous kernel in the stream completes (the kernel waits for it with
// griddepcontrol.wait before touching device memory).
template <typename K, typename... A>
cudaError_t launch_dependent(K kernel, unsigned blocks, unsigned threads, size_t smem, cudaStream_t st, const A&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}

template <typename S, int EQ, int VEC, int WARPS, int MINB>
cudaError_t launch_d2q9(const Params& P, cudaStream_t st) {
    const long long tiles = (long long)((P.nx + 32 * VEC - 1) / (32 * VEC)) * P.ny;
    const long long want = (tiles + WARPS - 1) / WARPS;   // at least one tile per warp
    const unsigned blocks = (unsigned)std::max(1ll, std::min(want, (long long)P.grid_blocks));
    return launch_dependent(k_collide_d2q9<S, EQ, VEC, WARPS, MINB>, blocks, 32 * WARPS, 0, st, P);
}

// Resident blocks per SM of a D2Q9 tile shape (occupancy calculator).
template <typename S, int EQ, int VEC, int WARPS, int MINB>
cudaError_t occupancy_d2q9(int* per_sm) {
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(per_sm, k_collide_d2q9<S, EQ, VEC, WARPS, MINB>,
                                                         32 * WARPS, 0);
}

template <typename S, int EQ, int R, int STAGES, int TX = kTmaTX>
cudaError_t launch_d2q9_tma(const Params& P, const void* tmap, cudaStream_t st) {
    constexpr size_t smem = tma_smem_bytes<S, R, STAGES, EQ, TX>();
    const long long tiles = (long long)((P.nx + TX - 1) / TX) * ((P.ny + R - 1) / R);
    const long long want = tiles;   // at least one tile per block
    const unsigned blocks = (unsigned)std::max(1ll, std::min(want, (long long)P.grid_blocks));
    return launch_dependent(k_collide_d2q9_tma<S, EQ, R, STAGES, TX>, blocks, 32 * R, smem, st, P,
                            *static_cast<const CUtensorMap*>(tmap));
}

template <typename S, int EQ, int R, int STAGES, int TX = kTmaTX>
cudaError_t setup_d2q9_tma(int* per_sm) {
    constexpr size_t smem = tma_smem_bytes<S, R, STAGES, EQ, TX>();
    cudaError_t e = cudaFuncSetAttribute(k_collide_d2q9_tma<S, EQ, R, STAGES, TX>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(per_sm, k_collide_d2q9_tma<S, EQ, R, STAGES, TX>,
                                                         32 * R, smem);
}

template <typename L, typename S, int EQ>
struct LaunchImpl {
    static cudaError_t collide(const Params& P, int shape, const void* tmap, cudaStream_t st) {
        if constexpr (L::Q == 9 && EQ >= EQ_ENERGY) {
            // the energy forms are built for two register-fed shapes (0: two
            // resident blocks, 128 registers per thread; 1-3: four, 64) and
            // two staged shapes (5: 6-row tiles, 168 registers; 4: 8-row
            // tiles, 128); shape 6 is refused for them by the host
            if (shape == 5) return launch_d2q9_tma<S, EQ, 6, 3>(P, tmap, st);
            if (shape == 4) return launch_d2q9_tma<S, EQ, 8, kStages8<S>>(P, tmap, st);
            if (shape == 0) return launch_d2q9<S, EQ, 1, 8, 2>(P, st);
            return launch_d2q9<S, EQ, 1, 8, 4>(P, st);
        } else if constexpr (L::Q == 9) {
            switch (shape) {
                case 1: return launch_d2q9<S, EQ, 1, 8, 4>(P, st);
                case 2: return launch_d2q9<S, EQ, 2, 8, 2>(P, st);
                case 3: return launch_d2q9<S, EQ, 4, 8, 1>(P, st);
                case 4: return launch_d2q9_tma<S, EQ, 8, kStages8<S>>(P, tmap, st);
                case 5: return launch_d2q9_tma<S, EQ, 6, 3>(P, tmap, st);
                case 6: return launch_d2q9_tma<S, EQ, 8, 2, 64>(P, tmap, st);
                default: return launch_d2q9<S, EQ, 1, 8, 3>(P, st);
            }
        } else {
            (void)shape;
            (void)tmap;
            const long long N = (long long)P.nx * P.ny;
            const unsigned blocks = (unsigned)((N + kSiteBlock - 1) / kSiteBlock);
            k_collide_site<L, S, EQ><<<blocks, kSiteBlock, 0, st>>>(P);
            return cudaGetLastError();
        }
    }
    // Many steps of a short D1Q3 run in one launch, from P.src to out;
    // cudaErrorNotSupported where the cluster does not serve the run.
    static cudaError_t tube(const Params& P, int steps, void* out, cudaStream_t st) {
        if constexpr (L::Q == 3) {
            const int per = (P.nx + kTubeBlocks - 1) / kTubeBlocks;
            if (per > kTubeThreads) return cudaErrorNotSupported;
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3(kTubeBlocks);
            cfg.blockDim = dim3((per + 31) / 32 * 32);
            cfg.dynamicSmemBytes = tube_smem_bytes<S>(P.nx);
            cfg.stream = st;
            cudaLaunchAttribute attr[1];
            attr[0].id = cudaLaunchAttributeClusterDimension;
            attr[0].val.clusterDim.x = kTubeBlocks;
            attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
            cfg.attrs = attr;
            cfg.numAttrs = 1;
            return cudaLaunchKernelEx(&cfg, k_tube<S, EQ>, P, steps, out);
        } else {
            (void)P; (void)steps; (void)out; (void)st;
            return cudaErrorNotSupported;
        }
    }
    // Whether this device runs the cluster of k_tube for n sites.
    static cudaError_t tube_setup(int n, int* ok) {
        *ok = 0;
        if constexpr (L::Q == 3) {
            const int per = (n + kTubeBlocks - 1) / kTubeBlocks;
            if (per > kTubeThreads) return cudaSuccess;
            const size_t smem = tube_smem_bytes<S>(n);
            cudaError_t e = cudaFuncSetAttribute(k_tube<S, EQ>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
            if (e != cudaSuccess) return e;
            e = cudaFuncSetAttribute(k_tube<S, EQ>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)tube_smem_bytes<S>(kTubeBlocks * kTubeThreads));
            if (e != cudaSuccess) return e;
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3(kTubeBlocks);
            cfg.blockDim = dim3((per + 31) / 32 * 32);
            cfg.dynamicSmemBytes = smem;
            cudaLaunchAttribute attr[1];
            attr[0].id = cudaLaunchAttributeClusterDimension;
            attr[0].val.clusterDim.x = kTubeBlocks;
            attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
            cfg.attrs = attr;
            cfg.numAttrs = 1;
            e = cudaOccupancyMaxActiveClusters(ok, k_tube<S, EQ>, &cfg);
            if (e != cudaSuccess) {
                *ok = 0;
                (void)cudaGetLastError();
            }
        }
        return cudaSuccess;
    }
    static cudaError_t occupancy(int shape, int* per_sm) {
        *per_sm = 1;
        if constexpr (L::Q == 9 && EQ >= EQ_ENERGY) {
            if (shape == 5) return setup_d2q9_tma<S, EQ, 6, 3>(per_sm);
            if (shape == 4) return setup_d2q9_tma<S, EQ, 8, kStages8<S>>(per_sm);
            if (shape == 0) return occupancy_d2q9<S, EQ, 1, 8, 2>(per_sm);
            return occupancy_d2q9<S, EQ, 1, 8, 4>(per_sm);
        } else if constexpr (L::Q == 9) {
            switch (shape) {
                case 1: return occupancy_d2q9<S, EQ, 1, 8, 4>(per_sm);
                case 2: return occupancy_d2q9<S, EQ, 2, 8, 2>(per_sm);
                case 3: return occupancy_d2q9<S, EQ, 4, 8, 1>(per_sm);
                case 4: return setup_d2q9_tma<S, EQ, 8, kStages8<S>>(per_sm);
                case 5: return setup_d2q9_tma<S, EQ, 6, 3>(per_sm);
                case 6: return setup_d2q9_tma<S, EQ, 8, 2, 64>(per_sm);
                default: return occupancy_d2q9<S, EQ, 1, 8, 3>(per_sm);
            }
        }
        return cudaSuccess;
    }
    static cudaError_t select(const Params& P, int stage_cap, int mode, cudaStream_t st) {
        const size_t smem = (size_t)stage_cap * (sizeof(unsigned long long) + sizeof(unsigned));
        k_select<L, S, EQ><<<1, kSelectThreads, smem, st>>>(P, stage_cap, mode);
        return cudaGetLastError();
    }
    static cudaError_t init_eq(const Params& P, const double* rho, const double* ux,
                               const double* uy, const double* e2, cudaStream_t st) {
        const long long N = (long long)P.nx * P.ny;
        k_init_eq<L, S, EQ><<<(unsigned)((N + 255) / 256), 256, 0, st>>>(P, rho, ux, uy, e2);
        return cudaGetLastError();
    }
    static cudaError_t import_state(const Params& P, const double* f, int i0, int i1, cudaStream_t st) {
        const long long N = (long long)P.nx * P.ny;
        if (i0 < 0 || i1 > L::Q || i0 >= i1 || N <= 0) return cudaErrorInvalidValue;
        k_import<L, S><<<(unsigned)((N + 255) / 256), 256, 0, st>>>(P, f, i0, i1);
        return cudaGetLastError();
    }
    static cudaError_t export_state(const Params& P, int mode, double* o0, double* o1, double* o2,
                                    double* o3, long long s0, long long s1, cudaStream_t st) {
        const long long N = (long long)P.nx * P.ny;
        if (s0 < 0 || s1 > N || s0 >= s1) return cudaErrorInvalidValue;
        k_export<L, S, EQ><<<(unsigned)((s1 - s0 + 255) / 256), 256, 0, st>>>(P, mode, o0, o1, o2, o3, s0, s1);
        return cudaGetLastError();
    }
    static cudaError_t ghost(const Params& P, void* field, int col, int right, void* buf, int dir,
                             cudaStream_t st) {
        const int n = 3 * P.ny;
        k_ghost<S><<<(n + 255) / 256, 256, 0, st>>>(P, static_cast<S*>(field), col, right, static_cast<S*>(buf),
                                                   dir);
        return cudaGetLastError();
    }
    static cudaError_t set_smem(int stage_cap) {
        const size_t smem = (size_t)stage_cap * (sizeof(unsigned long long) + sizeof(unsigned));
        return cudaFuncSetAttribute(k_select<L, S, EQ>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)smem);
    }
    static Launchers get() {
        Launchers l;
        l.collide = &collide;
        l.select = &select;
        l.init_eq = &init_eq;
        l.import_state = &import_state;
        l.export_state = &export_state;
        l.set_smem = &set_smem;
        l.ghost = &ghost;
        l.occupancy = &occupancy;
        l.tube = &tube;
        l.tube_setup = &tube_setup;
        return l;
    }
};

// Polynomial and entropic (mass and momentum) equilibria of one storage
// type; the energy forms are instantiated in their own translation units.
template <typename S>
Launchers launchers_basic(int lattice, int eq) {
    if (lattice == 0) {
        if (eq == EQ_POLY) return LaunchImpl<D1Q3, S, EQ_POLY>::get();
        return LaunchImpl<D1Q3, S, EQ_ENTROPIC>::get();
    }
    if (eq == EQ_POLY) return LaunchImpl<D2Q9, S, EQ_POLY>::get();
    return LaunchImpl<D2Q9, S, EQ_ENTROPIC>::get();
}

template <typename S>
Launchers launchers_energy(int eq) {
    if (eq == EQ_ENERGY_MLP) return LaunchImpl<D2Q9, S, EQ_ENERGY_MLP>::get();
    return LaunchImpl<D2Q9, S, EQ_ENERGY>::get();
}

}  // namespace lbm
