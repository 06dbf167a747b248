// Device-side physics of the two-population compressible lattice Boltzmann
// step (Sec. II C of the paper): equilibria, correction terms, collision,
// Grad's approximation (Sec. III A), blended-mesh kinematics (Sec. II A, II D)
// and the rigid-body RK4 (Sec. III B).  Templated on the arithmetic type R
// (double for the FP64 path, float for the FP32 path).
#pragma once

#include <cuda_runtime.h>
#include "lbfsi_internal.h"

namespace lbfsi {

// D2Q9 velocity of index q: 0:(0,0) 1:(1,0) 2:(0,1) 3:(-1,0) 4:(0,-1)
// 5:(1,1) 6:(-1,1) 7:(-1,-1) 8:(1,-1).  Resolved at compile time in unrolled loops.
__host__ __device__ constexpr int cxq(int q) {
    return (q == 1 || q == 5 || q == 8) ? 1 : ((q == 3 || q == 6 || q == 7) ? -1 : 0);
}
__host__ __device__ constexpr int cyq(int q) {
    return (q == 2 || q == 5 || q == 6) ? 1 : ((q == 4 || q == 7 || q == 8) ? -1 : 0);
}

// Reciprocal and square root in the precision of the path: the hardware
// approximations (relative error about 2^-23) on the float path.
__device__ __forceinline__ float rcp_(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
// (float64: the hardware's seed of about 20 bits and two Newton steps
// r += r (1 - x r), which square its error twice, to far below an ulp, the last
// with one rounding: 1/x correctly rounded but for values within some 2^-20 ulp
// of a tie.  For normal x whose reciprocal is normal; zero, infinity and NaN give
// NaN, which every caller treats as it does an infinity: a state of rho = 0 is
// non-physical and a departure solve with no determinant lost, by comparisons
// that NaN fails too.  The division costs 2 to 3.5% of a step: 80.1 -> 82.9 us on
// 96 x 96 x 3, 102.5 -> 106.2 on a 97 x 161 C-grid)
__host__ __device__ __forceinline__ double rcp_(double x) {
#ifdef __CUDA_ARCH__
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
    r = fma(r, fma(-x, r, 1.0), r);
    r = fma(r, fma(-x, r, 1.0), r);
    return r;
#else
    return 1.0 / x;
#endif
}
__device__ __forceinline__ float sqrt_(float x) {
    float y;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ double sqrt_(double x) { return sqrt(x); }
__device__ __forceinline__ float abs_(float x) { return fabsf(x); }
__device__ __forceinline__ double abs_(double x) { return fabs(x); }
// Arithmetic with its rounding fixed: the compiler neither fuses nor splits
// these, so an expression written with them rounds the same way in every
// kernel it is inlined into (a Newton iterate then converges to the same
// last bit whatever the tile shape or launch form).  The step kernels, whose
// instantiations have to step a node alike, are compiled without contraction
// (build.py), so the functions they share write their fused operations out.
__device__ __forceinline__ float fma_rn(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double fma_rn(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float add_rn(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ double add_rn(double a, double b) { return __dadd_rn(a, b); }
__host__ __device__ __forceinline__ float fm(float a, float b, float c) { return fmaf(a, b, c); }
__host__ __device__ __forceinline__ double fm(double a, double b, double c) { return fma(a, b, c); }

template <typename R>
struct Macro {
    R rho, ux, uy, T, E;
};

// The end of the kernel before in the stream, with its writes visible (nothing
// of a kernel launched by launch_behind may read or write global memory
// before); then the kernel behind may start (and wait in turn).
__device__ __forceinline__ void wait_previous() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// rho = sum f, rho u = sum f c, 2 rho E = sum g, T = (E - u^2/2) / Cv.
template <typename R>
__device__ __forceinline__ Macro<R> moments(const R* f, const R* g, R iCv) {
    const R rho = (f[0] + ((f[1] + f[3]) + (f[2] + f[4]))) + ((f[5] + f[7]) + (f[6] + f[8]));
    const R s2 = (g[0] + ((g[1] + g[3]) + (g[2] + g[4]))) + ((g[5] + g[7]) + (g[6] + g[8]));
    const R d = f[5] - f[7], e = f[6] - f[8];
    const R jx = (f[1] - f[3]) + (d - e), jy = (f[2] - f[4]) + (d + e);
    Macro<R> m;
    const R ir = rcp_(rho);
    m.rho = rho;
    m.ux = jx * ir;
    m.uy = jy * ir;
    m.E = R(0.5) * s2 * ir;
    m.T = fm(R(-0.5), fm(m.ux, m.ux, m.uy * m.uy), m.E) * iCv;
    return m;
}

// Product-form equilibrium f_i^eq = rho Phi_{cx}(u_x) Phi_{cy}(u_y) (Eq. feq).
template <typename R>
__host__ __device__ __forceinline__ void f_equilibrium(R rho, R ux, R uy, R T, R* f) {
    const R ax = fm(ux, ux, T), ay = fm(uy, uy, T);
    R px[3] = {R(0.5) * (ax - ux), R(1) - ax, R(0.5) * (ax + ux)};   // index c+1
    R py[3] = {R(0.5) * (ay - uy), R(1) - ay, R(0.5) * (ay + uy)};
#pragma unroll
    for (int c = 0; c < 3; ++c) px[c] *= rho;
#pragma unroll
    for (int q = 0; q < 9; ++q) f[q] = px[cxq(q) + 1] * py[cyq(q) + 1];
}

// W_i (z + q.c + A:(c c - T I)/(2T^2)) with the weights W of T: z the zeroth
// moment, q the first over T, A the second (the Hermite expansions of g and
// of the non-equilibrium parts); the last term takes five values (rest,
// x-axis, y-axis and the two diagonal pairs).
template <typename R>
__host__ __device__ __forceinline__ void hermite(R T, R iT, R z, R qx, R qy, R axx, R axy, R ayy, R* g) {
    const R iT2 = iT * iT, i2 = R(0.5) * iT2, A = axx + ayy, TA = T * A;
    const R w0 = R(0.5) * T, w1 = R(1) - T, Wa = w0 * w1, Wd = w0 * w0;
    g[0] = w1 * w1 * fm(-TA, i2, z);
    const R gx = Wa * fm(axx - TA, i2, z), gy = Wa * fm(ayy - TA, i2, z);
    g[1] = fm(Wa, qx, gx); g[3] = fm(-Wa, qx, gx); g[2] = fm(Wa, qy, gy); g[4] = fm(-Wa, qy, gy);
    const R gd = Wd * fm(A - TA, i2, z), t = axy * iT2;
    const R gp = fm(Wd, t, gd), gm = fm(-Wd, t, gd), sp = qx + qy, sm = qx - qy;
    g[5] = fm(Wd, sp, gp); g[7] = fm(-Wd, sp, gp); g[8] = fm(Wd, sm, gm); g[6] = fm(-Wd, sm, gm);
}

// g = W_i (2 rho E + q.c/T + (R^eq - 2 rho E T I):(c c - T I)/(2T^2)) + Psi_i
// (Eqs. geq, gstar).  H = E + T (energy flux of the enthalpy), R^eq as printed,
// Psi_i = B_i . X with B_0 = (1,1), B_{1,3} = (-1/2,0), B_{2,4} = (0,-1/2).
template <typename R>
__host__ __device__ __forceinline__ void g_hermite(R rho, R ux, R uy, R T, R E, R qx, R qy, R* g) {
    const R uxx = ux * ux, uyy = uy * uy, p = rho * T, e2 = R(2) * rho * E;
    const R e4 = fm(R(4), p, e2), pT = R(2) * p * T, iT = rcp_(T);
    // A = R^eq - 2 rho E T I
    hermite(T, iT, e2, qx * iT, qy * iT, fm(uxx, e4, pT), ux * uy * e4, fm(uyy, e4, pT), g);
    const R pre = rho * fm(R(-3), T, R(1)) * iT, tE = fm(R(2), T, E), TT = T * T;
    const R Xx = pre * fm(uxx, tE, TT), Xy = pre * fm(uyy, tE, TT), hx = R(0.5) * Xx, hy = R(0.5) * Xy;
    g[0] += Xx + Xy;
    g[1] -= hx;
    g[3] -= hx;
    g[2] -= hy;
    g[4] -= hy;
}

template <typename R>
__host__ __device__ __forceinline__ void g_equilibrium(R rho, R ux, R uy, R T, R Cv, R* g) {
    const R E = fm(Cv, T, R(0.5) * fm(ux, ux, uy * uy));
    const R H2 = R(2) * rho * (E + T);
    g_hermite(rho, ux, uy, T, E, H2 * ux, H2 * uy, g);
}

// Lane-wise arithmetic on (f_q, g_q) pairs: packed FP32x2 instructions on the
// float path (one instruction for both populations of a direction).
__device__ __forceinline__ float2 padd(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 pmul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 pfma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 psub(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.f, -1.f), a); }
__device__ __forceinline__ double2 padd(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 pmul(double2 a, double2 b) { return make_double2(a.x * b.x, a.y * b.y); }
__device__ __forceinline__ double2 pfma(double2 a, double2 b, double2 c) {
    return make_double2(fma(a.x, b.x, c.x), fma(a.y, b.y, c.y));
}
__device__ __forceinline__ double2 psub(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ float2 pair(float a, float b) { return make_float2(a, b); }
__device__ __forceinline__ double2 pair(double a, double b) { return make_double2(a, b); }

// What the collision of a node needs of its populations and relaxes them to.
// q* = q^eq + 2 u.(P - P^eq); 1/w = 1/2 + mu/(rho T dt), 1/w1 = 1/2 +
// (1/w - 1/2)/Pr.  g^qe differs from g^eq only in the heat flux, and
//   w (g^eq - g) + (w1 - w)(g^qe - g) = w1 (g' - g)
// for the g' of the one Hermite expansion with the flux q^eq + (1 - w/w1)
// (q* - q^eq), so one relaxation serves both; its (R^eq - 2 rho E T I):
// (c c - T I)/(2T^2) term takes five values (rest, x-axis, y-axis and the two
// diagonal pairs).
template <typename R>
struct Collision {
    R rho, e2, ux, uy, T, E, p, ax, ay, uxx, uyy, uxy, w, w1, iT, qx, qy;   // q: that flux over T
    template <typename R2>
    __device__ __forceinline__ void moments(const R2* p_, R mu, R muP, R dt, R iCv) {
        // opposite directions in pairs: their sums give rho, 2 rho E and P,
        // their differences rho u
        const R2 a = padd(p_[1], p_[3]), b = padd(p_[2], p_[4]), c = padd(p_[5], p_[7]), d = padd(p_[6], p_[8]);
        const R2 e = padd(c, d), s = padd(padd(p_[0], a), padd(b, e));
        rho = s.x;
        e2 = s.y;
        const R d5 = p_[5].x - p_[7].x, d6 = p_[6].x - p_[8].x;
        const R jx = (p_[1].x - p_[3].x) + (d5 - d6), jy = (p_[2].x - p_[4].x) + (d5 + d6);
        const R ir = rcp_(rho);
        ux = jx * ir;
        uy = jy * ir;
        E = R(0.5) * e2 * ir;
        uxx = ux * ux;
        uyy = uy * uy;
        uxy = ux * uy;
        T = fm(R(-0.5), uxx + uyy, E) * iCv;
        p = rho * T;
        ax = uxx + T;
        ay = uyy + T;
        // w = p dt / (p dt / 2 + mu), w1 with mu / Pr; 1 - w/w1 = (mu - mu/Pr) / (p dt / 2 + mu)
        const R pd = p * dt, rA = rcp_(fm(R(0.5), pd, mu));
        w = pd * rA;
        w1 = pd * rcp_(fm(R(0.5), pd, muP));
        const R dxx = fm(-rho, ax, a.x + e.x), dyy = fm(-rho, ay, b.x + e.x), dxy = fm(-rho, uxy, c.x - d.x);
        iT = rcp_(T);
        const R H2 = fm(R(2), p, e2) * iT, r = R(2) * iT * ((mu - muP) * rA);
        qx = fm(H2, ux, r * fm(ux, dxx, uy * dxy));
        qy = fm(H2, uy, r * fm(ux, dxy, uy * dyy));
    }
    __device__ __forceinline__ void f_target(R* f) const {
        const R hr = R(0.5) * rho;
        const R x0 = rho * (R(1) - ax), x1 = hr * (ax + ux), x3 = hr * (ax - ux);
        const R y0 = R(1) - ay, y1 = R(0.5) * (ay + uy), y3 = R(0.5) * (ay - uy);
        f[0] = x0 * y0; f[1] = x1 * y0; f[3] = x3 * y0; f[2] = x0 * y1; f[4] = x0 * y3;
        f[5] = x1 * y1; f[6] = x3 * y1; f[7] = x3 * y3; f[8] = x1 * y3;
    }
    __device__ __forceinline__ void g_target(R* g) const {
        const R iT2 = iT * iT, i2 = R(0.5) * iT2;
        const R e4 = fm(R(4), p, e2), pT = R(2) * p * T;
        const R axx = fm(uxx, e4, pT), ayy = fm(uyy, e4, pT), A = axx + ayy, TA = T * A;
        const R pre = rho * fm(R(-3), T, R(1)) * iT, tE = fm(R(2), T, E), TT = T * T;
        const R Xx = pre * fm(uxx, tE, TT), Xy = pre * fm(uyy, tE, TT);
        const R w0 = R(0.5) * T, w1_ = R(1) - T, Wa = w0 * w1_, Wd = w0 * w0;
        g[0] = fm(w1_ * w1_, fm(-TA, i2, e2), Xx + Xy);
        const R gx = fm(Wa, fm(axx - TA, i2, e2), R(-0.5) * Xx), gy = fm(Wa, fm(ayy - TA, i2, e2), R(-0.5) * Xy);
        g[1] = fm(Wa, qx, gx); g[3] = fm(-Wa, qx, gx); g[2] = fm(Wa, qy, gy); g[4] = fm(-Wa, qy, gy);
        const R gd = Wd * fm(A - TA, i2, e2), t = uxy * e4 * iT2;
        const R gp = fm(Wd, t, gd), gm = fm(-Wd, t, gd), sp = qx + qy, sm = qx - qy;
        g[5] = fm(Wd, sp, gp); g[7] = fm(-Wd, sp, gp); g[8] = fm(Wd, sm, gm); g[6] = fm(-Wd, sm, gm);
    }
};

// Collision at one node (Eq. f_boltz) on its (f_q, g_q) pairs p[9]: f* = f +
// w (f^eq - f) + dt phi, g* = g + w (g^eq - g) + (w1 - w)(g^qe - g), phi_i =
// -(1/2) c_i . Y on the axis velocities.  muP = mu / Pr, iCv = 1 / Cv.
template <typename R, typename R2>
__device__ __forceinline__ void collide_pairs(R2* p, R Yx, R Yy, R mu, R muP, R dt, R iCv) {
    Collision<R> c;
    c.moments(p, mu, muP, dt, iCv);
    R fe[9], ge[9];
    c.f_target(fe);
    c.g_target(ge);
    const R2 om = pair(c.w, c.w1);
    R2 d[9];
#pragma unroll
    for (int q = 0; q < 9; ++q) d[q] = pmul(om, psub(pair(fe[q], ge[q]), p[q]));
    if constexpr (sizeof(R) == 4) {
        // The relaxation leaves mass, momentum and energy unchanged in exact
        // arithmetic (sum f^eq = rho, sum f^eq c = rho u, sum g' = 2 rho E).
        // In float the rounded targets miss that by an ulp, and
        // at a node whose state barely changes the miss has the same sign at
        // every step, so it accumulates.  Its sums over the small changes are
        // exact to far below the populations' ulp: take them out of the rest
        // population (mass, energy) and of the axis pairs (momentum; their
        // sum, hence the mass, unchanged).
        const R2 e = padd(padd(padd(d[1], d[3]), padd(d[2], d[4])), padd(padd(d[5], d[7]), padd(d[6], d[8])));
        const R d5 = d[5].x - d[7].x, d6 = d[6].x - d[8].x;
        const R ex = R(0.5) * ((d[1].x - d[3].x) + (d5 - d6)), ey = R(0.5) * ((d[2].x - d[4].x) + (d5 + d6));
        d[0] = pmul(e, pair(R(-1), R(-1)));   // (d[0] minus the sum with d[0])
        d[1].x -= ex;
        d[3].x += ex;
        d[2].x -= ey;
        d[4].x += ey;
    }
    // dt phi on the axis velocities
    const R hyx = R(0.5) * dt * Yx, hyy = R(0.5) * dt * Yy;
    d[1].x -= hyx;
    d[3].x += hyx;
    d[2].x -= hyy;
    d[4].x += hyy;
#pragma unroll
    for (int q = 0; q < 9; ++q) p[q] = padd(p[q], d[q]);
}

// Grad's approximation at wall targets (Sec. III A, Eqs. fnoneq, gnoneq,
// strainrate): f = f^eq + dt f1, g = g^eq + dt g1.  gr: the gradients (d_x u_x,
// d_y u_x, d_x u_y, d_y u_y, d_x T, d_y T).
template <typename R>
struct WallTarget {
    R rho, ux, uy, T, gr[6];
};
// P^(1) of the targets (over dt): xx, xy, yy.
template <typename R>
__device__ __forceinline__ void grad_p1(const WallTarget<R>& t, R iom, R iCv, R* p1) {
    const R cP = -iom * t.rho * t.T, dv = (t.gr[0] + t.gr[3]) * iCv;
    p1[0] = cP * fm(R(2), t.gr[0], -dv);
    p1[1] = cP * (t.gr[2] + t.gr[1]);
    p1[2] = cP * fm(R(2), t.gr[3], -dv);
}
template <typename R>
__device__ __forceinline__ void grad_f(const WallTarget<R>& t, R mu, R dt, R iCv, R* f) {
    const R iom = fm(mu, rcp_(t.rho * t.T * dt), R(0.5));   // 1/omega
    R p1[3], h[9];
    grad_p1(t, iom, iCv, p1);
    f_equilibrium(t.rho, t.ux, t.uy, t.T, f);
    hermite(t.T, rcp_(t.T), R(0), R(0), R(0), p1[0], p1[1], p1[2], h);
#pragma unroll
    for (int q = 0; q < 9; ++q) f[q] = fm(dt, h[q], f[q]);
}
template <typename R>
__device__ __forceinline__ void grad_g(const WallTarget<R>& t, R mu, R dt, R Cv, R iCv, R iPr, R* g) {
    const R tau = mu * rcp_(t.rho * t.T * dt), iom = tau + R(0.5), iom1 = fm(tau, iPr, R(0.5));   // 1/omega, 1/omega_1
    const R ux = t.ux, uy = t.uy, T = t.T;
    R p1[3], h[9];
    grad_p1(t, iom, iCv, p1);
    const R E = fm(Cv, T, R(0.5) * fm(ux, ux, uy * uy)), iT = rcp_(T);
    const R dEx = fm(Cv, t.gr[4], fm(ux, t.gr[0], uy * t.gr[2])), dEy = fm(Cv, t.gr[5], fm(ux, t.gr[1], uy * t.gr[3]));
    const R cR = R(-2) * iom1 * t.rho * T, cq = cR * (Cv + R(1)), EpT = fm(R(2), T, E);
    const R qx = fm(cq, t.gr[4], R(2) * fm(ux, p1[0], uy * p1[1])), qy = fm(cq, t.gr[5], R(2) * fm(ux, p1[1], uy * p1[2]));
    const R rxx = cR * R(2) * fm(t.gr[0], EpT, ux * dEx), ryy = cR * R(2) * fm(t.gr[3], EpT, uy * dEy);
    const R rxy = cR * fm(t.gr[2] + t.gr[1], EpT, fm(ux, dEy, dEx * uy));
    g_equilibrium(t.rho, ux, uy, T, Cv, g);
    hermite(T, iT, R(0), qx * iT, qy * iT, rxx, rxy, ryy, h);
#pragma unroll
    for (int q = 0; q < 9; ++q) g[q] = fm(dt, h[q], g[q]);
}
template <typename R>
__device__ __forceinline__ void grad_populations(R rho, R ux, R uy, R T, R dudx, R dudy, R dvdx,
                                                 R dvdy, R dTdx, R dTdy, R mu, R dt, R Cv, R iCv, R iPr,
                                                 R* f, R* g) {
    const WallTarget<R> t{rho, ux, uy, T, {dudx, dudy, dvdx, dvdy, dTdx, dTdy}};
    grad_f(t, mu, dt, iCv, f);
    grad_g(t, mu, dt, Cv, iCv, iPr, g);
}

// Rotation part of a body state: sin(alpha) and cos(alpha) - 1 written as
// -2 sin^2(alpha/2) (no cancellation for small angles).  A state without
// rotation (every state of a transverse body) takes no transcendental call:
// sin(+-0) = +-0 exactly, so the values are the same.
struct BodyRot {
    double sa, cm1;
};
__host__ __device__ inline BodyRot body_rot(double alpha) {
    double sa = alpha, h = 0.5 * alpha;
    if (alpha != 0.0) {
        sa = sin(alpha);
        h = sin(0.5 * alpha);
    }
    return BodyRot{sa, -2.0 * h * h};
}

// Blended rigid map of one body (Sec. II D) for one body state s with
// previous state sp:  d(X) = A (X - Xp) + t with A = R(alpha) - I,
// t = (0, h);  x = X + (1 - r_blend) d(X).  The va.., vt. fields are the
// (state - previous state) differences times inv_dt, for V_G.
__host__ __device__ inline BodyMap<double> make_body_map(const BodyDev& b, const BodyStateDev& s,
                                                         BodyRot rs, const BodyStateDev& sp,
                                                         BodyRot rp, double inv_dt) {
    BodyMap<double> m;
    m.active = b.dof != 0;
    m.xc = b.xc; m.yc = b.yc; m.xp = b.xp; m.yp = b.yp;
    m.r_in = b.r_in;
    m.inv_w = b.inv_w;
    m.a00 = rs.cm1; m.a01 = -rs.sa; m.a10 = rs.sa; m.a11 = rs.cm1;
    m.tx = 0.0; m.ty = s.h;
    m.va00 = (rs.cm1 - rp.cm1) * inv_dt; m.va01 = -(rs.sa - rp.sa) * inv_dt;
    m.va10 = (rs.sa - rp.sa) * inv_dt; m.va11 = (rs.cm1 - rp.cm1) * inv_dt;
    m.vtx = 0.0; m.vty = (s.h - sp.h) * inv_dt;
    return m;
}

__host__ __device__ inline BodyMap<float> to_float(const BodyMap<double>& d) {
    BodyMap<float> m;
    m.active = d.active;
    m.xc = (float)d.xc; m.yc = (float)d.yc; m.xp = (float)d.xp; m.yp = (float)d.yp;
    m.r_in = (float)d.r_in; m.inv_w = (float)d.inv_w;
    m.a00 = (float)d.a00; m.a01 = (float)d.a01; m.a10 = (float)d.a10; m.a11 = (float)d.a11;
    m.tx = (float)d.tx; m.ty = (float)d.ty;
    m.va00 = (float)d.va00; m.va01 = (float)d.va01; m.va10 = (float)d.va10; m.va11 = (float)d.va11;
    m.vtx = (float)d.vtx; m.vty = (float)d.vty;
    return m;
}

// F = dx/dX of the blended map (analytic, includes the gradient of the blend
// factor) and V_G at absolute position (X, Y).  Outside the blended region
// F = I and V_G = 0 exactly, and the result is false.
template <typename R>
__device__ __forceinline__ bool kinematics(const BodyMap<R>& bm, R X, R Y, R& F00, R& F01, R& F10,
                                           R& F11, R& vx, R& vy) {
    F00 = R(1); F01 = R(0); F10 = R(0); F11 = R(1); vx = R(0); vy = R(0);
    if (!bm.active) return false;
    const R dx = X - bm.xc, dy = Y - bm.yc;
    const R dist = sqrt_(fm(dx, dx, dy * dy));
    const R s = (dist - bm.r_in) * bm.inv_w;
    if (s > R(1)) return false;
    R w, drx = R(0), dry = R(0);
    if (s < R(0)) {
        w = R(1);
    } else {
        // r5 = s^3 (10 - 15 s + 6 s^2), dr5/ds = 30 s^2 (1 - s)^2
        const R t = s * (R(1) - s);
        w = fm(-(s * s * s), fm(s, fm(R(6), s, R(-15)), R(10)), R(1));
        const R gq = R(30) * t * t * bm.inv_w * rcp_(dist);
        drx = gq * dx;
        dry = gq * dy;
    }
    const R px = X - bm.xp, py = Y - bm.yp;
    const R ux = fm(bm.a00, px, fm(bm.a01, py, bm.tx));
    const R uy = fm(bm.a10, px, fm(bm.a11, py, bm.ty));
    F00 = fm(-ux, drx, fm(w, bm.a00, R(1)));
    F01 = fm(-ux, dry, w * bm.a01);
    F10 = fm(-uy, drx, w * bm.a10);
    F11 = fm(-uy, dry, fm(w, bm.a11, R(1)));
    vx = w * fm(bm.va00, px, fm(bm.va01, py, bm.vtx));
    vy = w * fm(bm.va10, px, fm(bm.va11, py, bm.vty));
    return true;
}

// Kinematics of several bodies' blended maps: the displacements add
// (Sec. II D), so F = I + sum_b (F_b - I) and V_G = sum_b V_b; a body whose
// blended region does not hold the point adds nothing.
template <typename R>
__device__ __forceinline__ bool kinematics_sum(const BodyMap<R>* bm, int nb, R X, R Y, R& F00, R& F01,
                                               R& F10, R& F11, R& vx, R& vy) {
    bool moved = kinematics(bm[0], X, Y, F00, F01, F10, F11, vx, vy);
    for (int b = 1; b < nb; ++b) {
        R g00, g01, g10, g11, wx, wy;
        if (!kinematics(bm[b], X, Y, g00, g01, g10, g11, wx, wy)) continue;
        if (moved) {
            F00 += g00 - R(1); F01 += g01; F10 += g10; F11 += g11 - R(1);
            vx += wx; vy += wy;
        } else {
            F00 = g00; F01 = g01; F10 = g10; F11 = g11; vx = wx; vy = wy;
        }
        moved = true;
    }
    return moved;
}

// Fill a maps record: collision map from S_cur, stream maps from
// (S_next, S_vgprev); the float maps are the float64 ones rounded.
__host__ __device__ inline void build_maps(const BodyDev& b, const BodyStateDev& S_cur,
                                           const BodyStateDev& S_next,
                                           const BodyStateDev& S_vgprev, double dt, StepMaps& m) {
    m.S_cur = S_cur;
    m.S_next = S_next;
    m.S_vgprev = S_vgprev;
    const double inv_dt = 1.0 / dt;
    const BodyRot rc = body_rot(S_cur.alpha), rn = body_rot(S_next.alpha), rp = body_rot(S_vgprev.alpha);
    m.Kd = make_body_map(b, S_cur, rc, S_cur, rc, inv_dt);
    m.Sd = make_body_map(b, S_next, rn, S_vgprev, rp, inv_dt);
    m.Kf = to_float(m.Kd);
    m.Sf = to_float(m.Sd);
}

// Classical RK4 of the body ODE over dt with the load (Fx, Fy, M) held fixed
// (Sec. III B; weak coupling of Sec. III), for step n (from n dt to (n+1) dt).
// A pitch-plunge body in its forcing interval (Sec. IV D) has the pitch
// prescribed, alpha = amp sin(w_a t): the plunge row is integrated with the
// prescribed pitch acceleration at the stage times and alpha, alpha' are set
// to their values at (n+1) dt.
__host__ __device__ inline BodyStateDev rk4_body(const BodyDev& b, BodyStateDev s, double fy,
                                                 double mz, double dt, long long n) {
    if (b.dof == 2 && (double)(n + 1) * dt <= b.t_forced) {
        const double w = b.w_a, amp = b.pitch_amp;
        auto acc = [&](double t, double h, double v) {
            const double acc_a = -amp * w * w * sin(w * t);
            return (fy - b.k_h * h - b.s_a * acc_a) / b.m;
        };
        const double t0 = (double)n * dt, tm = ((double)n + 0.5) * dt, t1 = (double)(n + 1) * dt;
        const double h0 = s.h, v0 = s.hdot;
        const double k1h = v0, k1v = acc(t0, h0, v0);
        const double k2h = v0 + 0.5 * dt * k1v, k2v = acc(tm, h0 + 0.5 * dt * k1h, v0 + 0.5 * dt * k1v);
        const double k3h = v0 + 0.5 * dt * k2v, k3v = acc(tm, h0 + 0.5 * dt * k2h, v0 + 0.5 * dt * k2v);
        const double k4h = v0 + dt * k3v, k4v = acc(t1, h0 + dt * k3h, v0 + dt * k3v);
        s.h = h0 + dt / 6.0 * (k1h + 2.0 * k2h + 2.0 * k3h + k4h);
        s.hdot = v0 + dt / 6.0 * (k1v + 2.0 * k2v + 2.0 * k3v + k4v);
        s.alpha = amp * sin(w * t1);
        s.adot = amp * w * cos(w * t1);
        return s;
    }
    if (b.dof == 1) {
        auto acc = [&](double h, double v) { return (fy - b.k * h - b.c * v) / b.m; };
        const double h0 = s.h, v0 = s.hdot;
        const double k1h = v0, k1v = acc(h0, v0);
        const double k2h = v0 + 0.5 * dt * k1v, k2v = acc(h0 + 0.5 * dt * k1h, v0 + 0.5 * dt * k1v);
        const double k3h = v0 + 0.5 * dt * k2v, k3v = acc(h0 + 0.5 * dt * k2h, v0 + 0.5 * dt * k2v);
        const double k4h = v0 + dt * k3v, k4v = acc(h0 + dt * k3h, v0 + dt * k3v);
        s.h = h0 + dt / 6.0 * (k1h + 2.0 * k2h + 2.0 * k3h + k4h);
        s.hdot = v0 + dt / 6.0 * (k1v + 2.0 * k2v + 2.0 * k3v + k4v);
    } else if (b.dof == 2) {
        const double det = b.m * b.i_a - b.s_a * b.s_a;
        auto accel = [&](const double* y, double* a) {
            const double r0 = fy - b.k_h * y[0], r1 = mz - b.k_a * y[1];
            a[0] = (b.i_a * r0 - b.s_a * r1) / det;
            a[1] = (-b.s_a * r0 + b.m * r1) / det;
        };
        double y0[4] = {s.h, s.alpha, s.hdot, s.adot}, k[4][4], yt[4], acc2[2];
        for (int st = 0; st < 4; ++st) {
            const double c = (st == 0) ? 0.0 : (st == 3 ? 1.0 : 0.5);
            for (int n = 0; n < 4; ++n) yt[n] = y0[n] + (st ? c * dt * k[st - 1][n] : 0.0);
            accel(yt, acc2);
            k[st][0] = yt[2]; k[st][1] = yt[3]; k[st][2] = acc2[0]; k[st][3] = acc2[1];
        }
        double y1[4];
        for (int n = 0; n < 4; ++n)
            y1[n] = y0[n] + dt / 6.0 * (k[0][n] + 2.0 * k[1][n] + 2.0 * k[2][n] + k[3][n]);
        s.h = y1[0]; s.alpha = y1[1]; s.hdot = y1[2]; s.adot = y1[3];
    }
    return s;
}

}  // namespace lbfsi
