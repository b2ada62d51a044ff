// lbm_energy.cuh -- entropic quasiequilibrium with the energy constraint
// (D2Q9): the maximiser of the perfect entropy S = -sum f ln(f/W) ((PerfEnt))
// subject to m(f) = M = (rho, rho u1, rho u2, 2E) ((argmax)).  Its Lagrange
// form (Sec. 3.3) is ln(f*_i / W_i) = mu . (1, v_x, v_y, |v|^2).  The
// weights are products of the one-dimensional weights (2/3, 1/6, 1/6) and
// |v|^2 = v_x^2 + v_y^2, so f* factorises: f*_i = rho p_x(v_x) p_y(v_y) with
//   p(+-1) = (P +- u) / 2,  p(0) = 1 - P,
// u the axis's velocity and P its second moment.  Three of the four
// constraints hold by this form and P_x + P_y = T = 2E / rho; what is left
// of the Lagrange form is that both axes have the same energy multiplier
// mu_3 = ln c,
//   (P_x^2 - u_x^2) / (1 - P_x)^2 = (P_y^2 - u_y^2) / (1 - P_y)^2 = c^2 / 4.
// With tau = T / 2, P_x = tau + e, P_y = tau - e, a = 1 - tau this is one
// cubic in e,
//   h(e) = 4 e^3 - D e^2 + 2 a (T - S) e - D a^2 = 0,
//   D = u_x^2 - u_y^2,  S = u_x^2 + u_y^2,
// whose root in the realisable range (every p > 0) is unique (the dual is
// strictly convex) and has h' > 0.
//
// The solve has two phases.  FP32: Newton on the energy multiplier from its
// start point (0, the polynomial start, or the network's prediction), on
// F(mu_3) = P_x + P_y - T with, k2 = c^2 / 4 and w = sqrt(k2 + u^2 (1 - k2)),
//   P = (u^2 + k2) / (k2 + w),  dP/dmu_3 = (P^2 - u^2) / w.
// It gives e = (P_x - P_y) / 2, corrected to first order for the multiplier's
// last step d; the error left, about |D| d^2 / 3, stops the iteration at 1e-6.
// Then Newton steps on h with h in float-float (FP32 / FP16 storage) or FP64
// (FP64 storage) and the slope in FP32: a step d leaves at most
// |12 e - D| d^2 / h' + 4e-7 |d|, and the steps end when that bound on the
// error of P (the residual max |m(f*) - M| / rho of the energy condition) is
// at or below 1e-12 (FP64: the caller's stop).
//
// The former solve was Newton on all three multipliers (three exponentials,
// a 3 x 3 covariance and its Cholesky factors per iteration, residual sums
// of nine float-float terms): bound by FP32 issue at about 2000 instructions
// per site.  2048 x 1024, FP32: 64 us per step against 166 us
// (three such runs side by side; one alone 89 us against 205 us), 49 us with
// two sites per lane in packed arithmetic.
#pragma once

#include "lbm_device.cuh"

namespace lbm {

constexpr int kNewton32Max = 16;
constexpr int kNewton64Max = 6;
constexpr float kNewton32Tol = 1e-6f;    // |D| d^2 at which the FP32 phase stops
constexpr double kNewtonTol = 1e-12;

struct NewtonCount {
    unsigned it32, it64, sites, fails;
    __device__ __forceinline__ void add(const NewtonCount& o) {
        it32 += o.it32;
        it64 += o.it64;
        sites += o.sites;
        fails += o.fails;
    }
};

__device__ __forceinline__ float sqrt_approx(float x) {
    float r;
    asm("sqrt.approx.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

__device__ __forceinline__ float rcp_approx(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ f2 rcp_approx(f2 x) { return f2(rcp_approx(x.x), rcp_approx(x.y)); }
__device__ __forceinline__ f2 sqrt_approx(f2 x) { return f2(sqrt_approx(x.x), sqrt_approx(x.y)); }

// One evaluation of F at k2: the multiplier's Newton step d and e corrected
// for it to first order (F: float, or f2 for a pair of sites).
template <typename F>
__device__ __forceinline__ void energy_newton32(F u2x, F u2y, F T, F k2, F& d, F& e) {
    const F one = F(1.0f) - k2;
    const F wx = sqrt_approx(dfma<F>(u2x, one, k2)), wy = sqrt_approx(dfma<F>(u2y, one, k2));
    const F Px = (u2x + k2) * rcp_approx(k2 + wx), Py = (u2y + k2) * rcp_approx(k2 + wy);
    const F dx = (Px * Px - u2x) * rcp_approx(wx), dy = (Py * Py - u2y) * rcp_approx(wy);
    d = ((Px + Py) - T) * rcp_approx(dx + dy);
    e = F(0.5f) * ((Px - Py) - (dx - dy) * d);
}

// The FP32 phase: e = (P_x - P_y) / 2 for u_x, u_y, T from the start point
// mu3 of the energy multiplier.  u2x, u2y: u_x^2, u_y^2.
__device__ __forceinline__ float energy_phase32(float u2x, float u2y, float T, float mu3, NewtonCount& nc) {
    const float D = fabsf(u2x - u2y);
    float k2 = 0.25f * __expf(2.0f * mu3);
    unsigned it = 0;
    float e;
    for (;; it++) {
        float d;
        energy_newton32<float>(u2x, u2y, T, k2, d, e);
        if (!(D * (d * d) > kNewton32Tol || fabsf(d) > 0.5f) || it == kNewton32Max) break;
        d = fminf(fmaxf(d, -0.5f), 0.5f);   // far start points: damped
        k2 *= __expf(-2.0f * d);
    }
    nc.it32 += it;
    return e;
}

// Bound on the error of e that a step d of the finishing phase leaves.
__device__ __forceinline__ float energy_step_error(float e, float D, float islope, float d) {
    return fmaf(fabsf(fmaf(12.0f, e, -D)) * islope * d, d, 4e-7f * fabsf(d));
}

// Energy-constrained quasiequilibrium f*_i (FP64) of one site from rho,
// u and th = 2E / rho; mu3: start point of the energy multiplier.  FP64 steps
// continue until the error of e is at or below stop_tol (1e-12, or closer to
// the rounding floor for FP64 storage).  Returns false if it did not reach
// 1e-12 or no positive f* has these moments (the site then keeps the last
// iterate).  mu (optional): the solution's multipliers mu_1 .. mu_3 in FP64.
// GB300's FP64 pipe is slow (two operations per SM and clock), so only the
// cubic, the factors and their products are FP64: about 50 operations.
__device__ __forceinline__ bool energy_solve(double rho, double ux, double uy, double th, float mu3, double* fstar,
                                             NewtonCount& nc, float stop_tol, double* mu = nullptr) {
    const float uxf = (float)ux, uyf = (float)uy, Tf = (float)th;
    const float u2x = uxf * uxf, u2y = uyf * uyf;
    double e = (double)energy_phase32(u2x, u2y, Tf, mu3, nc);
    const double D = (ux - uy) * (ux + uy), S = fma(ux, ux, uy * uy);
    const double tau = 0.5 * th, a = 1.0 - tau;
    const double c1 = (a + a) * (th - S), c0 = D * a * a;
    const float Df = u2x - u2y, c1f = (2.0f - Tf) * (Tf - (u2x + u2y));
    float left = INFINITY;
    int it = 0;
    while (it < kNewton64Max) {
        const float ef = (float)e;
        const float islope = recip<float>(fmaf(fmaf(12.0f, ef, -2.0f * Df), ef, c1f));
        const double h = fma(fma(fma(4.0, e, -D), e, c1), e, -c0);
        const double d = h * (double)islope;
        e -= d;
        it++;
        left = energy_step_error(ef, Df, islope, (float)d);
        if (!(left > stop_tol)) break;
    }
    nc.it64 += (unsigned)it;
    nc.sites += 1u;
    const double Px = tau + e, Py = tau - e;
    const bool ok = left <= (float)kNewtonTol && Px > fabs(ux) && Py > fabs(uy) && Px < 1.0 && Py < 1.0;
    if (!ok) nc.fails += 1u;
    const double h2 = 0.5 * rho;
    const double x0 = rho * (1.0 - Px), xp = h2 * (Px + ux), xm = h2 * (Px - ux);
    const double y0 = 1.0 - Py, yp = 0.5 * (Py + uy), ym = 0.5 * (Py - uy);
    fstar[0] = x0 * y0;
    fstar[1] = xp * y0;
    fstar[2] = x0 * yp;
    fstar[3] = xm * y0;
    fstar[4] = x0 * ym;
    fstar[5] = xp * yp;
    fstar[6] = xm * yp;
    fstar[7] = xm * ym;
    fstar[8] = xp * ym;
    if (mu) {
        const double q = (Px - ux) * (Px + ux);
        mu[0] = 0.5 * log((Px + ux) / (Px - ux));
        mu[1] = 0.5 * log((Py + uy) / (Py - uy));
        mu[2] = 0.5 * log(4.0 * q / ((1.0 - Px) * (1.0 - Px)));
    }
    return ok;
}

// ---------------------------------------------------------------------------
// Float-float arithmetic: a value is the unevaluated sum hi + lo of two
// floats with |lo| <= ulp(hi) / 2 (about 48 significant bits).  Built on the
// error-free transformations two-sum (Knuth) and two-product (by one fused
// multiply-add); the addition is the "sloppy" form of Dekker's algorithm
// (its error is relative to |a| + |b|, which is what the residual sums
// below need).  The library is compiled without multiply-add contraction,
// so every rounding written here happens as written.
// ---------------------------------------------------------------------------
template <typename F>
struct ff_of {
    F hi, lo;
};
using ff = ff_of<float>;
using ffp = ff_of<f2>;   // a pair of sites, packed

template <typename F>
__device__ __forceinline__ ff_of<F> ff_fast_two_sum(F a, F b) {   // |a| >= |b| or a == 0
    const F s = a + b;
    return {s, b - (s - a)};
}
template <typename F>
__device__ __forceinline__ ff_of<F> ff_two_sum(F a, F b) {
    const F s = a + b;
    const F bb = s - a;
    return {s, (a - (s - bb)) + (b - bb)};
}
template <typename F>
__device__ __forceinline__ ff_of<F> ff_add(ff_of<F> a, ff_of<F> b) {
    const ff_of<F> s = ff_two_sum(a.hi, b.hi);
    return ff_fast_two_sum(s.hi, s.lo + (a.lo + b.lo));
}
template <typename F>
__device__ __forceinline__ ff_of<F> ff_sub(ff_of<F> a, ff_of<F> b) {   // the operations of a + (-b)
    const F s = a.hi - b.hi;
    const F bb = s - a.hi;
    return ff_fast_two_sum(s, ((a.hi - (s - bb)) - (b.hi + bb)) + (a.lo - b.lo));
}
template <typename F>
__device__ __forceinline__ ff_of<F> ff_scale(ff_of<F> a, float p2) {   // p2 a power of two
    return {a.hi * F(p2), a.lo * F(p2)};
}
template <typename F>
__device__ __forceinline__ ff_of<F> ff_mul(ff_of<F> a, ff_of<F> b) {
    const F p = a.hi * b.hi;
    F e = dfma<F>(a.hi, b.hi, -p);
    e = dfma<F>(a.hi, b.lo, e);
    e = dfma<F>(a.lo, b.hi, e);
    return ff_fast_two_sum(p, e);
}
template <typename F>
__device__ __forceinline__ ff_of<F> ff_mul_f(ff_of<F> a, F b) {
    const F p = a.hi * b;
    F e = dfma<F>(a.hi, b, -p);
    e = dfma<F>(a.lo, b, e);
    return ff_fast_two_sum(p, e);
}
// 1 / a: an FP32 reciprocal r plus one Newton-Raphson correction r (1 - a r),
// whose leading part fma(-a.hi, r, 1) is exact.
__device__ __forceinline__ float ff_seed(float x) { return __frcp_rn(x); }
__device__ __forceinline__ f2 ff_seed(f2 x) { return f2(__frcp_rn(x.x), __frcp_rn(x.y)); }
template <typename F>
__device__ __forceinline__ ff_of<F> ff_recip(ff_of<F> a) {
    const F r = ff_seed(a.hi);
    F e = dfma<F>(-a.hi, r, F(1.0f));
    e = dfma<F>(-a.lo, r, e);
    return ff_fast_two_sum(r, r * e);
}
// a + b and a - b where |a.hi| >= |b.hi| (or a = 0): the leading sum's error
// by the fast two-sum.
template <typename F>
__device__ __forceinline__ ff_of<F> ff_add_ord(ff_of<F> a, ff_of<F> b) {
    const ff_of<F> s = ff_fast_two_sum(a.hi, b.hi);
    return ff_fast_two_sum(s.hi, s.lo + (a.lo + b.lo));
}
template <typename F>
__device__ __forceinline__ ff_of<F> ff_sub_ord(ff_of<F> a, ff_of<F> b) {   // the operations of a + (-b)
    const F s = a.hi - b.hi;
    return ff_fast_two_sum(s, ((a.hi - s) - b.hi) + (a.lo - b.lo));
}

// What the float-float finish needs besides e, from the FP32 moments.
template <typename F>
struct EnergyFinish {
    ff_of<F> ux, uy, T, D, c1, c0, tau;

    __device__ __forceinline__ EnergyFinish(F rho, F jx, F jy, F e2, F& u2x, F& u2y) {
        const F zero = F(0.0f);
        const ff_of<F> one = {F(1.0f), zero}, ir = ff_recip(ff_of<F>{rho, zero});
        ux = ff_mul_f(ir, jx);
        uy = ff_mul_f(ir, jy);
        T = ff_mul_f(ir, e2);
        const ff_of<F> xx = ff_mul(ux, ux), yy = ff_mul(uy, uy);
        u2x = xx.hi;
        u2y = yy.hi;
        D = ff_sub(xx, yy);
        const ff_of<F> S = ff_add(xx, yy);
        tau = ff_scale(T, 0.5f);
        const ff_of<F> a = ff_sub_ord(one, tau);
        c1 = ff_scale(ff_mul(a, ff_sub_ord(T, S)), 2.0f);
        c0 = ff_mul(ff_mul(a, a), D);
    }
    // Newton step d at e, with its slope's reciprocal
    __device__ __forceinline__ F step(ff_of<F> e, F& islope) const {
        islope = recip<F>(dfma<F>(dfma<F>(F(12.0f), e.hi, F(-2.0f) * D.hi), e.hi, c1.hi));
        ff_of<F> h = ff_mul(ff_sub(ff_scale(e, 4.0f), D), e);
        h = ff_sub(ff_mul(ff_add(h, c1), e), c0);
        return h.hi * islope;
    }
    // The deviations gs_i = f*_i - W_i; Px, Py (leading parts) out.
    __device__ __forceinline__ void factors(ff_of<F> e, F rho, F* gs, F& px, F& py) const {
        const ff_of<F> one = {F(1.0f), F(0.0f)};
        const ff_of<F> Px = ff_add_ord(tau, e), Py = ff_sub_ord(tau, e);
        px = Px.hi;
        py = Py.hi;
        const F half = F(0.5f) * rho;
        const ff_of<F> x[3] = {ff_mul_f(ff_sub_ord(one, Px), rho), ff_mul_f(ff_add_ord(Px, ux), half),
                               ff_mul_f(ff_sub_ord(Px, ux), half)};
        const ff_of<F> y[3] = {ff_sub_ord(one, Py), ff_scale(ff_add_ord(Py, uy), 0.5f),
                               ff_scale(ff_sub_ord(Py, uy), 0.5f)};
#pragma unroll
        for (int i = 0; i < 9; i++) {
            const ff_of<F> f = ff_mul(x[D2Q9::cx(i) < 0 ? 2 : D2Q9::cx(i)], y[D2Q9::cy(i) < 0 ? 2 : D2Q9::cy(i)]);
            constexpr float whi[3] = {(float)(4.0 / 9.0), (float)(1.0 / 9.0), (float)(1.0 / 36.0)};
            constexpr float wlo[3] = {(float)(4.0 / 9.0 - (double)(float)(4.0 / 9.0)),
                                      (float)(1.0 / 9.0 - (double)(float)(1.0 / 9.0)),
                                      (float)(1.0 / 36.0 - (double)(float)(1.0 / 36.0))};
            const int k = i == 0 ? 0 : (i < 5 ? 1 : 2);
            gs[i] = (f.hi - F(whi[k])) + (f.lo - F(wlo[k]));
        }
    }
};

// Energy-constrained quasiequilibrium for FP32 / FP16 storage from the FP32
// moments (rho, j, 2E): the FP32 phase, then Newton steps on h with h in
// float-float until the error of e is at or below 1e-12; the factors and
// their products in float-float.  Writes the deviations gs_i = f*_i - W_i
// (these forms have rho0 = 1), whose leading difference is exact while f*_i
// is within a factor two of W_i.  Returns false if the error did not reach
// 1e-12 or no positive f* has these moments (the site keeps the last
// iterate).  The ordered additions below have |a| >= |b| for every
// realisable state: T > S, tau < 1, |e| < tau, P > |u|.
__device__ __forceinline__ bool energy_solve_ff(float rho, float jx, float jy, float e2, float mu3, float* gs,
                                                NewtonCount& nc) {
    float u2x, u2y, px, py;
    const EnergyFinish<float> E(rho, jx, jy, e2, u2x, u2y);
    ff e = {energy_phase32(u2x, u2y, E.T.hi, mu3, nc), 0.0f};
    float left = INFINITY;
    int it = 0;
    while (it < kNewton64Max) {
        float islope;
        const float d = E.step(e, islope);
        left = energy_step_error(e.hi, E.D.hi, islope, d);
        e = ff_sub(e, ff{d, 0.0f});
        it++;
        if (!(left > (float)kNewtonTol)) break;
    }
    nc.it64 += (unsigned)it;
    nc.sites += 1u;
    E.factors(e, rho, gs, px, py);
    const bool ok = left <= (float)kNewtonTol && px > fabsf(E.ux.hi) && py > fabsf(E.uy.hi) && px < 1.0f && py < 1.0f;
    if (!ok) nc.fails += 1u;
    return ok;
}

// The same for a pair of sites in packed arithmetic, every operation the
// scalar one's half by half: a site that is done keeps its iterate while the
// other goes on.  nc: the two sites' counts (they are added up only for the
// sites that are the caller's).  2048 x 1024, FP32, three runs side by side: 55 ->
// 50 us per step.
__device__ __forceinline__ void energy_solve_pair(f2 rho, f2 jx, f2 jy, f2 e2, f2 mu3, f2* gs, NewtonCount* nc) {
    f2 u2x, u2y, px, py;
    const EnergyFinish<f2> E(rho, jx, jy, e2, u2x, u2y);
    // FP32 phase
    const f2 d2 = u2x - u2y;
    const float Dx = fabsf(d2.x), Dy = fabsf(d2.y);
    f2 k2 = f2(0.25f) * f2(__expf(2.0f * mu3.x), __expf(2.0f * mu3.y)), e0;
    for (unsigned it = 0;; it++) {
        f2 d;
        energy_newton32<f2>(u2x, u2y, E.T.hi, k2, d, e0);
        const bool gx = (Dx * (d.x * d.x) > kNewton32Tol || fabsf(d.x) > 0.5f) && it < kNewton32Max;
        const bool gy = (Dy * (d.y * d.y) > kNewton32Tol || fabsf(d.y) > 0.5f) && it < kNewton32Max;
        if (!(gx || gy)) break;
        if (gx) {
            k2.x *= __expf(-2.0f * fminf(fmaxf(d.x, -0.5f), 0.5f));
            nc[0].it32 += 1u;
        }
        if (gy) {
            k2.y *= __expf(-2.0f * fminf(fmaxf(d.y, -0.5f), 0.5f));
            nc[1].it32 += 1u;
        }
    }
    // float-float finish
    ffp e = {e0, f2(0.0f)};
    float lx = INFINITY, ly = INFINITY;
    for (int it = 0; it < kNewton64Max; it++) {
        f2 islope;
        f2 d = E.step(e, islope);
        const bool gx = lx > (float)kNewtonTol, gy = ly > (float)kNewtonTol;   // (still to go)
        if (gx) {
            lx = energy_step_error(e.hi.x, E.D.hi.x, islope.x, d.x);
            nc[0].it64 += 1u;
        } else {
            d.x = 0.0f;
        }
        if (gy) {
            ly = energy_step_error(e.hi.y, E.D.hi.y, islope.y, d.y);
            nc[1].it64 += 1u;
        } else {
            d.y = 0.0f;
        }
        e = ff_sub(e, ffp{d, f2(0.0f)});
        if (!(lx > (float)kNewtonTol) && !(ly > (float)kNewtonTol)) break;
    }
    E.factors(e, rho, gs, px, py);
    nc[0].sites += 1u;
    nc[1].sites += 1u;
    if (!(lx <= (float)kNewtonTol && px.x > fabsf(E.ux.hi.x) && py.x > fabsf(E.uy.hi.x) && px.x < 1.0f && py.x < 1.0f))
        nc[0].fails += 1u;
    if (!(ly <= (float)kNewtonTol && px.y > fabsf(E.ux.hi.y) && py.y > fabsf(E.uy.hi.y) && px.y < 1.0f && py.y < 1.0f))
        nc[1].fails += 1u;
}

}  // namespace lbm
