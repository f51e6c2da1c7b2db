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
// warp-wide FMA whose three operands are vector registers every 68 clocks (at
// 2.07 GHz, 152 SMs busy), but an add, a multiply, or an FMA with a literal,
// constant-bank or uniform-register operand only every 80.6; every large FP64
// path here is bound by that unit.  So the constants are kept in vector
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

// min(num/den, 1) for num, den nonzero with the same sign.  When
// |num| >= |den| the quotient rounds to >= 1, so the division is skipped.
template <typename R>
__device__ __forceinline__ R limited_ratio(R num, R den)
{
    const auto mag = ~(decltype(fbits(num)))0 >> 1;
    return (fbits(num) & mag) >= (fbits(den) & mag) ? R(1) : Fp<R>::div(num, den);
}

// Limited states at the interface between cells a (left) and b (right)
// (Eqs. Pratio, limitleft, limitright): the ratio at cell a is
// (pb - pa)/(pa - pam) and gives QL = Qa + min(ratio, 1)/2 (Qb - Qa) when it
// lies in (0, inf); the inverse ratio at cell b, (pb - pa)/(pbp - pb), gives
// QR = Qb + min(inverse, 1)/2 (Qa - Qb); otherwise first order.
// lfirst / rfirst: the side was left first order (a copy of its cell).
template <typename R>
__device__ __forceinline__ void euler_reconstruct(const R qa[3], const R qb[3], R pam, R pa,
                                                  R pb, R pbp, R ql[3], R qr[3], bool& lfirst, bool& rfirst,
                                                  const Units<R>& k)
{
    using F = Fp<R>;
    R num = F::sub(pb, pa, k), den = F::sub(pa, pam, k);
    lfirst = !same_sign(num, den);
    if (!lfirst) {
        R h = F::mul(F::half(k), limited_ratio(num, den), k);
#pragma unroll
        for (int c = 0; c < 3; ++c) ql[c] = F::fma(h, F::sub(qb[c], qa[c], k), qa[c]);
    } else {
#pragma unroll
        for (int c = 0; c < 3; ++c) ql[c] = qa[c];
    }
    R num2 = F::sub(pbp, pb, k);
    rfirst = !same_sign(num2, num);
    if (!rfirst) {
        R h = F::mul(F::half(k), limited_ratio(num, num2), k);
#pragma unroll
        for (int c = 0; c < 3; ++c) qr[c] = F::fma(h, F::sub(qa[c], qb[c], k), qb[c]);
    } else {
#pragma unroll
        for (int c = 0; c < 3; ++c) qr[c] = qb[c];
    }
}

// G = 2 Flux from the limited states: F(QR) + F(QL) + r_sp (QL - QR), with
// F(Q) = (rho u, rho u^2 + P, u (E + P)) (Eq. EulerF) and spectral radius
// r_sp = sqrt(gamma (gamma-1) (e_sp - u_sp^2/2)) + |u_sp| from sqrt(rho)-weighted
// Roe averages of u and of e = E/rho (gamma P_sp / rho_sp with
// P_sp = (gamma-1) rho_sp (e_sp - u_sp^2/2)).  Divisions by rho and by the
// weight sum are multiplications by correctly rounded reciprocals.
//
// Per-cell values are reused.  Where the limiter leaves a side first order
// (uniform regions: the pressure difference is 0), the side state is its
// cell's state, and the flux's pressure, velocity, specific energy e = E/rho
// and sqrt(rho) of that side are the cell's own.  euler_cell forms them once
// per cell with exactly the operations a limited side's state gets, so
// reusing them gives the same bits.
template <typename R>
__device__ __forceinline__ R euler_cell(R r, R m, R E, R gm1, R& u, R& e, R& s, const Units<R>& k)
{
    R ir;
    const R p = euler_pressure(r, m, E, gm1, u, ir, k);
    e = Fp<R>::mul(E, ir, k);
    s = Fp<R>::sqrt(r);
    return p;
}

// Pressure, velocity, e and sqrt(rho) of a limited side state q.
template <typename R>
__device__ __forceinline__ R euler_side(const R q[3], R gm1, R& u, R& e, R& s, const Units<R>& k)
{
    return euler_cell(q[0], q[1], q[2], gm1, u, e, s, k);
}

// ca / cb: (u, e, sqrt(rho)) of cells a and b (as euler_cell forms them).
template <typename R>
__device__ __forceinline__ void euler_interface_cached(const R qa[3], const R qb[3], R pam, R pa, R pb,
                                                       R pbp, const R ca[3], const R cb[3], R gm1, R ggm1,
                                                       R G[3], const Units<R>& k)
{
    using F = Fp<R>;
    R ql[3], qr[3];
    bool lfirst, rfirst;
    euler_reconstruct(qa, qb, pam, pa, pb, pbp, ql, qr, lfirst, rfirst, k);
    R pl, ul, el, sl, pr, ur, er, sr;
    if (lfirst) {
        pl = pa;
        ul = ca[0];
        el = ca[1];
        sl = ca[2];
    } else {
        pl = euler_side(ql, gm1, ul, el, sl, k);
    }
    if (rfirst) {
        pr = pb;
        ur = cb[0];
        er = cb[1];
        sr = cb[2];
    } else {
        pr = euler_side(qr, gm1, ur, er, sr, k);
    }
    R fl1 = F::fma(ql[1], ul, pl);
    R fl2 = F::mul(ul, F::add(ql[2], pl, k), k);
    R fr1 = F::fma(qr[1], ur, pr);
    R fr2 = F::mul(ur, F::add(qr[2], pr, k), k);
    R iw = F::rcp(F::add(sl, sr, k));
    R usp = F::mul(F::fma(sl, ul, F::mul(sr, ur, k)), iw, k);
    R esp = F::mul(F::fma(sl, el, F::mul(sr, er, k)), iw, k);
    R c2 = F::mul(ggm1, F::fma(F::mul(F::mhalf(k), usp, k), usp, esp), k);
    R rsp = F::add(F::sqrt(c2), F::abs(usp), k);
    G[0] = F::fma(rsp, F::sub(ql[0], qr[0], k), F::add(qr[1], ql[1], k));
    G[1] = F::fma(rsp, F::sub(ql[1], qr[1], k), F::add(fr1, fl1, k));
    G[2] = F::fma(rsp, F::sub(ql[2], qr[2], k), F::add(fr2, fl2, k));
}

// Finite-volume RK2 stage: out = base - (h/dx)(Flux_{i+1/2} - Flux_{i-1/2})
// = fma(kh, G_{i+1/2} - G_{i-1/2}, base).
template <typename R>
__device__ __forceinline__ R euler_update(R gp, R gm, R base, R kh, const Units<R>& k)
{
    return Fp<R>::fma(kh, Fp<R>::sub(gp, gm, k), base);
}

}  // namespace swp
