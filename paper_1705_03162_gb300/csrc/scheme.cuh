// Point updates of the three test problems (arXiv:1705.03162, Appendices
// A-C), shared by the classic and the swept kernels so that both produce the
// same bits.  Every operation is an explicit round-to-nearest intrinsic, so
// the compiler neither contracts nor reorders: the rounding sequence is the
// one written here.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

namespace swp {

enum Eq : int { HEAT = 0, KS = 1, EULER = 2 };
enum Bc : int { PERIODIC = 0, REFLECTIVE = 1, DIRICHLET = 2 };

// Constants of the arithmetic below, each in a register of its own (see Fp).
template <typename R> struct Units {};
template <> struct Units<double> {
    double one, mone, m2, half, mhalf, nzero;   // 1, -1, -2, 1/2, -1/2, -0
};

// x in a vector register: the condition always holds, but the compiler cannot
// tell, nor that the lanes agree, so it keeps the value per lane.
__device__ __forceinline__ double per_lane(double x) { return threadIdx.x < blockDim.x ? x : 0.0; }
__device__ __forceinline__ float per_lane(float x) { return x; }

// The units equation EQ's point updates use.
template <typename R, int EQ>
__device__ __forceinline__ Units<R> make_units()
{
    Units<R> k{};
    if constexpr (sizeof(R) == 8) {
        k.one = per_lane(1.0);
        if constexpr (EQ == HEAT) k.m2 = per_lane(-2.0);
        if constexpr (EQ != HEAT) k.mone = per_lane(-1.0);
        if constexpr (EQ == EULER) {
            k.half = per_lane(0.5);
            k.mhalf = per_lane(-0.5);
            k.nzero = per_lane(-0.0);
        }
    }
    return k;
}

// The same as literals, which the compiler folds: for a kernel that waits on one
// dependent chain instead of filling the FP64 unit.
template <typename R> __device__ __forceinline__ Units<R> literal_units();
template <> __device__ __forceinline__ Units<float> literal_units<float>() { return {}; }
template <> __device__ __forceinline__ Units<double> literal_units<double>() { return {1.0, -1.0, -2.0, 0.5, -0.5, -0.0}; }

// Round-to-nearest arithmetic in the working precision.
//
// FP64 sums, differences and products are written as fused multiply-adds:
// a + b = fma(a, 1, b), a - b = fma(b, -1, a), a b = fma(a, b, -0), each rounded
// once, with the same bits (signed zeros included).  GB300's FP64 unit takes a
// warp-wide FMA whose three operands are vector registers every 64.0 clocks (the
// SM's own clock counter, all 152 SMs busy, 1 to 4 warps per sub-partition), but an
// add, a multiply, or an FMA with a literal, constant-bank or uniform-register operand
// only every 76.0; every large FP64 path here is bound by that unit.  So the constants are kept in vector
// registers whose value the compiler cannot see (Units).  Measured in G
// point-updates/s before and after: KS 2^20 swept 39.8 / 42.5, classic graph
// 29.6 / 33.6; heat 2^20 swept 169 / 188, 2^24 classic 169 / 195; Euler 2^20
// swept 3.66 / 3.90.
template <typename R> struct Fp;
template <> struct Fp<double> {
    using K = const Units<double>&;
    static __device__ __forceinline__ double add(double a, double b, K k) { return __fma_rn(a, k.one, b); }
    static __device__ __forceinline__ double sub(double a, double b, K k) { return __fma_rn(b, k.mone, a); }
    static __device__ __forceinline__ double mul(double a, double b, K k) { return __fma_rn(a, b, k.nzero); }
    static __device__ __forceinline__ double fma(double a, double b, double c) { return __fma_rn(a, b, c); }
    static __device__ __forceinline__ double m2(K k) { return k.m2; }
    static __device__ __forceinline__ double half(K k) { return k.half; }
    static __device__ __forceinline__ double mhalf(K k) { return k.mhalf; }
    static __device__ __forceinline__ double div(double a, double b) { return __ddiv_rn(a, b); }
    static __device__ __forceinline__ double rcp(double a) { return __drcp_rn(a); }
    static __device__ __forceinline__ double sqrt(double a) { return __dsqrt_rn(a); }
    static __device__ __forceinline__ double abs(double a) { return fabs(a); }
};
template <> struct Fp<float> {
    using K = const Units<float>&;
    static __device__ __forceinline__ float add(float a, float b, K) { return __fadd_rn(a, b); }
    static __device__ __forceinline__ float sub(float a, float b, K) { return __fsub_rn(a, b); }
    static __device__ __forceinline__ float mul(float a, float b, K) { return __fmul_rn(a, b); }
    static __device__ __forceinline__ float fma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
    static __device__ __forceinline__ float m2(K) { return -2.0f; }
    static __device__ __forceinline__ float half(K) { return 0.5f; }
    static __device__ __forceinline__ float mhalf(K) { return -0.5f; }
    static __device__ __forceinline__ float div(float a, float b) { return __fdiv_rn(a, b); }
    static __device__ __forceinline__ float rcp(float a) { return __frcp_rn(a); }
    static __device__ __forceinline__ float sqrt(float a) { return __fsqrt_rn(a); }
    static __device__ __forceinline__ float abs(float a) { return fabsf(a); }
};

// Per-problem constants, formed on the host in double and rounded once to R.
template <typename R> struct Coefs {
    R fo;                 // heat: Fourier number alpha dt / dx^2
    R a1[2], a4[2], beta[2], gam[2];  // KS stage s (0 predictor h = dt/2, 1 final h = dt):
                          // a1 = -h/(4dx), a4 = -h/dx^4, beta = a2 - 4 a4,
                          // gam = 6 a4 - 2 a2, a2 = -h/dx^2
    R kh[2];              // Euler stage s: -(h/dx)/2 (G below is twice the flux)
    R gm1, ggm1;          // gamma - 1, gamma (gamma - 1)
    R ghost_l[3], ghost_r[3];  // Dirichlet end states, conserved
};

// The constants a kernel's point updates use, in vector registers (Fp says why).
template <typename R, int EQ>
__device__ __forceinline__ Coefs<R> lane_coefs(const Coefs<R>& c)
{
    Coefs<R> o{};
    if constexpr (EQ == HEAT) o.fo = per_lane(c.fo);
#pragma unroll
    for (int s = 0; s < 2; ++s) {
        if constexpr (EQ == KS) {
            o.a1[s] = per_lane(c.a1[s]);
            o.a4[s] = per_lane(c.a4[s]);
            o.beta[s] = per_lane(c.beta[s]);
            o.gam[s] = per_lane(c.gam[s]);
        }
        if constexpr (EQ == EULER) o.kh[s] = per_lane(c.kh[s]);
    }
    if constexpr (EQ == EULER) {
        o.gm1 = per_lane(c.gm1);
        o.ggm1 = per_lane(c.ggm1);
    }
#pragma unroll
    for (int v = 0; v < 3; ++v) {
        o.ghost_l[v] = c.ghost_l[v];
        o.ghost_r[v] = c.ghost_r[v];
    }
    return o;
}

// ---------------------------------------------------------------------------
// Heat, FTCS (Appendix A, Eq. heatdisc):
//   T' = Fo (T_{i+1} + T_{i-1}) + (1 - 2 Fo) T_i = T_i + Fo (T_{i+1} - 2 T_i + T_{i-1})
// ---------------------------------------------------------------------------
template <typename R>
__device__ __forceinline__ R heat_point(R tm, R t0, R tp, R fo, const Units<R>& k)
{
    using F = Fp<R>;
    R lap = F::fma(F::m2(k), t0, F::add(tp, tm, k));
    return F::fma(fo, lap, t0);
}

// ---------------------------------------------------------------------------
// Kuramoto-Sivashinsky, one midpoint-RK2 stage (Appendix B, Eqs. KSDisc, RKm,
// RKf): out = base + h f(v), base = u^m, h = dt/2 (predictor) or dt (final).
// The Laplacian (1, -2, 1)/dx^2 and the fourth difference (1, -4, 6, -4, 1)/dx^4
// combine into one five-point stencil with weights a4 (v++, v--),
// beta = a2 - 4 a4 (v+, v-) and gam = 6 a4 - 2 a2 (v); the nonlinear term
// a1 (v+^2 - v-^2) = a1 (v+ - v-)(v+ + v-) shares the factor v+ + v-, so
//   h f = gam v + a4 (v++ + v--) + (beta + a1 (v+ - v-)) (v+ + v-),
// with a1 = -h/(4dx), a2 = -h/dx^2, a4 = -h/dx^4.  Seven FP operations; the
// dependent chain is three deep.
// ---------------------------------------------------------------------------
template <typename R>
__device__ __forceinline__ R ks_point(R vmm, R vm, R v0, R vp, R vpp, R base,
                                      R a1, R a4, R beta, R gam, const Units<R>& k)
{
    using F = Fp<R>;
    const R t = F::fma(a1, F::sub(vp, vm, k), beta);
    R acc = F::fma(gam, v0, base);
    acc = F::fma(a4, F::add(vpp, vmm, k), acc);
    return F::fma(t, F::add(vp, vm, k), acc);
}

// ---------------------------------------------------------------------------
// Euler (Appendix C).  Conserved Q = (rho, rho u, E), E total energy per volume.
// ---------------------------------------------------------------------------

// Velocity and pressure, Eq. EulerP: u = (rho u)/rho, P = (gamma-1)(E - (rho u) u / 2),
// dividing by rho as a multiplication by the correctly rounded 1/rho (ir).
template <typename R>
__device__ __forceinline__ R euler_pressure(R r, R m, R E, R gm1, R& u, R& ir, const Units<R>& k)
{
    using F = Fp<R>;
    ir = F::rcp(r);
    u = F::mul(m, ir, k);
    return F::mul(gm1, F::fma(F::mul(F::mhalf(k), m, k), u, E), k);
}

// Sign and magnitude tests on the IEEE bit patterns (integer pipe; GB300's
// FP64 pipe would spend a full slot on each comparison).  Equal to the
// floating-point comparisons for every non-NaN value.
__device__ __forceinline__ uint64_t fbits(double x) { return (uint64_t)__double_as_longlong(x); }
__device__ __forceinline__ uint32_t fbits(float x) { return (uint32_t)__float_as_uint(x); }

// (a > 0 && b > 0) || (a < 0 && b < 0): both nonzero, equal sign bits
template <typename R>
__device__ __forceinline__ bool same_sign(R a, R b)
{
    const auto ua = fbits(a), ub = fbits(b);
    constexpr int top = 8 * sizeof(R) - 1;
    return (ua << 1) != 0 && (ub << 1) != 0 && ((ua ^ ub) >> top) == 0;
}

// What a level keeps per cell beside its pressure.  The limiter (Eqs. Pratio,
// limitleft, limitright) compares the pressure differences on the two sides of
// a cell, and both states that the cell gives, QL = Q + min(ratio, 1)/2 (Q+ - Q) on
// its right and QR = Q + min(1/ratio, 1)/2 (Q- - Q) on its left, ratio =
// (p+ - p)/(p - p-), are limited or first order together: the ratio lies in
// (0, inf) exactly when both differences are nonzero with the same sign.
//  - first order (uniform regions, extrema): both states are the cell's own, so
//    its velocity, specific energy e = E/rho and sqrt(rho) serve both interfaces;
//  - limited: min(ratio, 1)/2 and min(1/ratio, 1)/2, of which one is 1/2 (a
//    quotient of |num| >= |den| rounds to at least 1), so one division serves both;
//    the third value is kLimited, which no sqrt yields.
// Against evaluating each interface side on its own this drops a division, and
// on limited cells the cell's own square root: 200000 cells limited everywhere,
// 100 steps, 9.93 to 8.34 ms.
constexpr uint64_t kLimitedBits = 0xbff0000000000000ull;   // -1.0

__device__ __forceinline__ bool euler_limited(double third) { return (uint64_t)__double_as_longlong(third) == kLimitedBits; }
__device__ __forceinline__ bool euler_limited(float third) { return third == -1.0f; }

// First pass: pressure, and the velocity and specific energy of a cell.
template <typename R>
__device__ __forceinline__ R euler_cell(R r, R m, R E, R gm1, R& u, R& e, const Units<R>& k)
{
    R ir;
    const R p = euler_pressure(r, m, E, gm1, u, ir, k);
    e = Fp<R>::mul(E, ir, k);
    return p;
}

// Second pass, with the pressures of the cell and its neighbours: c0, c1 hold
// (u, e) from the first pass and become, with c2, the cell's kept values.
// ROOT: c2 holds sqrt(r) already.
template <bool ROOT, typename R>
__device__ __forceinline__ void euler_limit(R pm, R p, R pp, R r, R& c0, R& c1, R& c2, const Units<R>& k)
{
    using F = Fp<R>;
    const R dp = F::sub(pp, p, k), dm = F::sub(p, pm, k);
    if (same_sign(dp, dm)) {
        const auto mag = ~(decltype(fbits(dp)))0 >> 1;
        const auto ap = fbits(dp) & mag, am = fbits(dm) & mag;
        const bool steep = ap >= am;   // ratio >= 1
        const R h = ap == am ? R(0.5) : F::mul(F::half(k), F::div(steep ? dm : dp, steep ? dp : dm), k);
        c0 = steep ? R(0.5) : h;
        c1 = steep ? h : R(0.5);
        c2 = R(-1);
    } else if (!ROOT) {
        c2 = F::sqrt(r);
    }
}

// One side of an interface: its state q (the cell's, or limited towards the
// other cell's state qo with factor h), velocity, e and sqrt(rho), and the flux
// F(q) = (rho u, f1, f2) = (rho u, rho u^2 + P, u (E + P)) (Eq. EulerF).
template <typename R>
__device__ __forceinline__ void euler_side(const R qc[3], const R qo[3], R pc, const R c[3], R h, R gm1, R q[3], R& f1,
                                           R& f2, R& u, R& e, R& s, const Units<R>& k)
{
    using F = Fp<R>;
    R p;
    if (euler_limited(c[2])) {
#pragma unroll
        for (int v = 0; v < 3; ++v) q[v] = F::fma(h, F::sub(qo[v], qc[v], k), qc[v]);
        p = euler_cell(q[0], q[1], q[2], gm1, u, e, k);
        s = F::sqrt(q[0]);
    } else {
#pragma unroll
        for (int v = 0; v < 3; ++v) q[v] = qc[v];
        p = pc;
        u = c[0];
        e = c[1];
        s = c[2];
    }
    f1 = F::fma(q[1], u, p);
    f2 = F::mul(u, F::add(q[2], p, k), k);
}

// G = 2 Flux from the two sides, F(QR) + F(QL) + r_sp (QL - QR), with spectral
// radius r_sp = sqrt(gamma (gamma-1) (e_sp - u_sp^2/2)) + |u_sp| from
// sqrt(rho)-weighted Roe averages of u and of e = E/rho (gamma P_sp / rho_sp with
// P_sp = (gamma-1) rho_sp (e_sp - u_sp^2/2)).  Divisions by rho and by the
// weight sum are multiplications by correctly rounded reciprocals.
// su, se: sr ur and sr er.
template <typename R>
__device__ __forceinline__ void euler_join(const R ql[3], R fl1, R fl2, R ul, R el, R sl, const R qr[3], R fr1, R fr2,
                                           R su, R se, R sr, R ggm1, R G[3], const Units<R>& k)
{
    using F = Fp<R>;
    R iw = F::rcp(F::add(sl, sr, k));
    R usp = F::mul(F::fma(sl, ul, su), iw, k);
    R esp = F::mul(F::fma(sl, el, se), iw, k);
    R c2 = F::mul(ggm1, F::fma(F::mul(F::mhalf(k), usp, k), usp, esp), k);
    R rsp = F::add(F::sqrt(c2), F::abs(usp), k);
    G[0] = F::fma(rsp, F::sub(ql[0], qr[0], k), F::add(qr[1], ql[1], k));
    G[1] = F::fma(rsp, F::sub(ql[1], qr[1], k), F::add(fr1, fl1, k));
    G[2] = F::fma(rsp, F::sub(ql[2], qr[2], k), F::add(fr2, fl2, k));
}

// Third pass, the interface between cells a (left) and b (right) with kept values
// ca and cb.
template <typename R>
__device__ __forceinline__ void euler_interface(const R qa[3], const R qb[3], R pa, R pb, const R ca[3], const R cb[3],
                                                R gm1, R ggm1, R G[3], const Units<R>& k)
{
    R ql[3], qr[3], fl1, fl2, ul, el, sl, fr1, fr2, ur, er, sr;
    euler_side(qa, qb, pa, ca, ca[0], gm1, ql, fl1, fl2, ul, el, sl, k);
    euler_side(qb, qa, pb, cb, cb[1], gm1, qr, fr1, fr2, ur, er, sr, k);
    euler_join(ql, fl1, fl2, ul, el, sl, qr, fr1, fr2, Fp<R>::mul(sr, ur, k), Fp<R>::mul(sr, er, k), sr, ggm1, G, k);
}

// Finite-volume RK2 stage: out = base - (h/dx)(Flux_{i+1/2} - Flux_{i-1/2})
// = fma(kh, G_{i+1/2} - G_{i-1/2}, base).
template <typename R>
__device__ __forceinline__ R euler_update(R gp, R gm, R base, R kh, const Units<R>& k)
{
    return Fp<R>::fma(kh, Fp<R>::sub(gp, gm, k), base);
}

}  // namespace swp
