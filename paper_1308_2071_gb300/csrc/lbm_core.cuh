// The collision of one node (or of two nodes side by side, V = F2) with as few
// operations as the model allows, for the FP32 and FP64 storage variants.
//
// The step is bound by instructions as soon as it is not bound by memory
// (FP64 always; FP32 in the batched, two-step and L2-resident cases), so the
// formulas of Eq. 16-23 and 27-36 are rearranged, equal in exact arithmetic:
//  - Eq. 22 makes u = j + F / 2 with F the total force of Eq. 4, so F = 2 (u -
//    j) needs no drag term of its own, the momentum gains exactly F per step
//    whatever s_3 and s_5 are, and the forcing moments (Eq. 19) are products
//    of u and u - j;
//  - Eq. 23 makes 6 dP and -9 dP combinations of the populations, so that the
//    energy moments enter through z = 4 b - a - |u|^2 / phi and the local mass
//    m_0 only (a, b: sums of the axis and of the diagonal populations);
//  - Eq. 36 makes n_0 - T a constant, so zeta_0 is immaterial and the source
//    (Eq. 30) adds w~_j Q / sigma to every population;
//  - the wall rule (Section 4) yields populations with the same properties
//    (their s18 and n_0 match the imposed p_b and T_b, and u_b - j_b = u_f -
//    j_f), so a wall node runs the same formulas with u = 0 and its own force.
// One node then takes 134 operations instead of 220 (FP64, uniform porosity).
// Measured, us per step before and after: FP64 1024^2 483 -> 317 (the FP64 unit
// bounds it either way), FP32 64^2 4.6 -> 3.1, 601 x 397 with a porosity field 6.7 ->
// 5.5, 1024^2 21 -> 18.6 (observation included).
//
// Every operation is an explicit round-to-nearest intrinsic, so the compiler
// fuses nothing on its own: each kernel, launch shape and precision of the
// index arithmetic gives the same bits for the same node.
//
// Collision in increments (f+ = f + M^-1 (m+ - m), g+ = g + N^-1 (n+ - n)): the
// rounded factors scale the change of a step only (see collide below for the
// bias that the direct form has in FP32).
#pragma once

#include "lbm_device.cuh"

namespace lbm {

// ---- explicit operations -----------------------------------------------------------

// Type of the constants that go with node values of type V.
template <class V> struct ScalarOf {
    using type = V;
};
template <> struct ScalarOf<F2> {
    using type = float;
};
template <class V> using Scalar = typename ScalarOf<V>::type;

namespace op {
// Two nodes at once: each is one paired instruction, rounded per node like its
// scalar counterpart, so both forms give the same bits.
__device__ __forceinline__ F2 add(F2 a, F2 b) { return F2(__fadd2_rn(a.v, b.v)); }
__device__ __forceinline__ F2 sub(F2 a, F2 b) { return F2(__ffma2_rn(b.v, make_float2(-1.f, -1.f), a.v)); }
__device__ __forceinline__ F2 mul(F2 a, F2 b) { return F2(__fmul2_rn(a.v, b.v)); }
__device__ __forceinline__ F2 fma(F2 a, F2 b, F2 c) { return F2(__ffma2_rn(a.v, b.v, c.v)); }
__device__ __forceinline__ F2 add(F2 a, float b) { return add(a, F2(b)); }
__device__ __forceinline__ F2 add(float a, F2 b) { return add(F2(a), b); }
__device__ __forceinline__ F2 sub(float a, F2 b) { return sub(F2(a), b); }
__device__ __forceinline__ F2 mul(float a, F2 b) { return mul(F2(a), b); }
__device__ __forceinline__ F2 fma(float a, F2 b, F2 c) { return fma(F2(a), b, c); }
__device__ __forceinline__ F2 fma(F2 a, float b, float c) { return fma(a, F2(b), F2(c)); }
__device__ __forceinline__ F2 fma(F2 a, float b, F2 c) { return fma(a, F2(b), c); }
__device__ __forceinline__ F2 fma(float a, F2 b, float c) { return fma(F2(a), b, F2(c)); }
__device__ __forceinline__ float add(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float sub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float mul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float fma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double add(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ double sub(double a, double b) { return __dsub_rn(a, b); }
__device__ __forceinline__ double mul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ double fma(double a, double b, double c) { return __fma_rn(a, b, c); }

// a b - c for an exact product a b
__device__ __forceinline__ float fms(float a, float b, float c) { return fma(a, b, -c); }
__device__ __forceinline__ double fms(double a, double b, double c) { return fma(a, b, -c); }
__device__ __forceinline__ F2 fms(float a, F2 b, F2 c) { return sub(mul(a, b), c); }

// sqrt(x) for x in the normal range (the callers add a floor far below any
// rounding): the hardware's reciprocal square root y, then, in FP32, one step of Newton's
// method for x - s^2 from s = x y, or, from its 20-bit FP64 form, the binomial series
// sqrt(x) = t (1 - e)^(-1/2) = t (1 + e/2 + 3 e^2 / 8 + ...) with t = x y and e = 1 - t y of
// the order of 2^-19.  Relative errors over the callers' arguments at most 1.0 x 2^-24, as a
// rounded root's, and 1.48 x 2^-53 (inverse: 1.63 x 2^-24 and 1.0 x 2^-53, inverse_full: 1.0).
__device__ __forceinline__ float root(float x) {
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    const float s = mul(x, y);
    return fma(fma(-s, s, x), mul(0.5f, y), s);
}
__device__ __forceinline__ double root(double x) {
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double t = mul(x, y), e = fma(-t, y, 1.0);
    return fma(t, mul(fma(0.375, e, 0.5), e), t);
}
__device__ __forceinline__ F2 root(F2 x) {
    float2 y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y.x) : "f"(x.v.x));
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y.y) : "f"(x.v.y));
    const F2 s = mul(x, F2(y));
    return fma(fma(mul(-1.f, s), s, x), mul(0.5f, F2(y)), s);
}
// 1 / x for normal x, in FP32 below 2^126 (above, the hardware gives 0; see velocity): the
// hardware's approximation, in FP64 with the first three terms of the geometric series
// 1 / x = y / (1 - e) = y (1 + e + e^2 + ...), e = 1 - x y of the order of 2^-19.
__device__ __forceinline__ float inverse(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ double inverse(double x) {
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double e = fma(-x, y, 1.0);
    return fma(y, fma(e, e, e), y);
}
__device__ __forceinline__ float minus_inverse(float x) { return inverse(-x); }
__device__ __forceinline__ double minus_inverse(double x) { return inverse(-x); }
__device__ __forceinline__ F2 minus_inverse(F2 x) { return F2(inverse(-x.v.x), inverse(-x.v.y)); }
__device__ __forceinline__ F2 inverse(F2 x) { return F2(inverse(x.v.x), inverse(x.v.y)); }
// 1 / phi of a porosity field: to the last bit or so (Newton's step in FP32)
__device__ __forceinline__ float inverse_full(float x) {
    const float y = inverse(x);
    return fma(y, fma(-x, y, 1.f), y);
}
__device__ __forceinline__ double inverse_full(double x) { return inverse(x); }
__device__ __forceinline__ F2 inverse_full(F2 x) { return F2(inverse_full(x.v.x), inverse_full(x.v.y)); }
// a, or b where a is larger; a NaN stays one
__device__ __forceinline__ float at_most(float a, float b) {
    float r;
    asm("min.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ F2 at_most(F2 a, float b) { return F2(at_most(a.v.x, b), at_most(a.v.y, b)); }
__device__ __forceinline__ double at_most(double a, double) { return a; }
// smallest |v|^2 that root() sees: sqrt(x + tiny) differs from sqrt(x) by less than 1e-18
__device__ __forceinline__ float tiny(float) { return 1e-37f; }
__device__ __forceinline__ double tiny(double) { return 1e-36; }
__device__ __forceinline__ F2 tiny(F2) { return F2(1e-37f); }
}  // namespace op

// ---- drag ----------------------------------------------------------------------------

// What Eq. 22 needs of a node's porosity: with cc = c_lin / 4 and l1 = c_quad /
// 2, ec = cc + cc^2, and hb = phi g beta / 2; iphi = 1 / phi.
//
// The uniform porosity's cc is held at kMostDrag in FP32 (fill_coef), where u is 1e-19
// of v, so that S + w, 2 cc^2, stays in the reciprocal's range (see velocity).
constexpr float kMostDrag = 4.6e18f;
template <class V> struct Por {
    V hb, cc, ec, l1, iphi;
};
template <class V, bool FIELD> __device__ __forceinline__ Por<V> por_of(const Coll<Scalar<V>>& k, V phi) {
    Por<V> p;
    if constexpr (FIELD) {
        const V ip = op::inverse_full(phi);
        const V om = op::sub(V(1), phi), t = op::mul(om, op::mul(ip, ip));
        p.hb = op::mul(k.hb, phi);
        p.cc = op::mul(op::mul(k.cc, om), t);
        p.ec = op::fma(p.cc, p.cc, p.cc);
        p.l1 = op::mul(k.l1, t);
        p.iphi = ip;
    } else {
        p.hb = V(k.hb);
        p.cc = V(k.cc);
        p.ec = V(k.ec);
        p.l1 = V(k.l1);
        p.iphi = V(k.iphi);
    }
    return p;
}

// ---- sums and macroscopic values -----------------------------------------------------

template <class V> struct Sums {
    V a, b, ex, ey, dx, dy, m7, m8;  // of the flow populations
    V tt, n0, n1, n2, n4;            // of the thermal populations
};

// n_0 (T - T0, or T - T0 - F framed, without the source half-step), in the
// one association used wherever a temperature is formed from pulled values.
template <class V> __device__ __forceinline__ V heat(const V (&h)[5]) {
    return op::add(h[0], op::add(op::add(h[1], h[3]), op::add(h[2], h[4])));
}

template <class V> __device__ __forceinline__ Sums<V> sums_of(const V (&d)[9], const V (&h)[5]) {
    Sums<V> s;
    const V a13 = op::add(d[1], d[3]), a24 = op::add(d[2], d[4]);
    const V s56 = op::add(d[5], d[6]), m56 = op::sub(d[5], d[6]);
    const V s78 = op::add(d[7], d[8]), m78 = op::sub(d[7], d[8]);
    s.ex = op::sub(d[1], d[3]);
    s.ey = op::sub(d[2], d[4]);
    s.a = op::add(a13, a24);
    s.m7 = op::sub(a13, a24);
    s.b = op::add(s56, s78);
    s.dy = op::sub(s56, s78);
    s.dx = op::sub(m56, m78);
    s.m8 = op::add(m56, m78);
    const V t13 = op::add(h[1], h[3]), t24 = op::add(h[2], h[4]);
    s.n1 = op::sub(h[1], h[3]);
    s.n2 = op::sub(h[2], h[4]);
    s.tt = op::add(t13, t24);
    s.n4 = op::sub(t13, t24);
    s.n0 = op::add(h[0], s.tt);
    return s;
}

template <class V> struct Vel {
    V ux, uy, dux, duy, vm, ngd;  // u, u - j, |v|, minus the fraction of v that the drag takes
    V S;                          // 1/2 + sqrt(l0^2 + l1 |v|)
    V dTl, dT;                    // T - T0 - F (framed storage; else T - T0) and T - T0
};

// Eq. 36, 22 and 21.  F: the node's frame (0 without frames).  u = v / (l0 +
// sqrt(l0^2 + l1 |v|)) as v - v g / (1 + g), with g / (1 + g) = w / (S + w), S =
// 1/2 + sqrt(1/4 + e), e = l0^2 + l1 |v| - 1/4, w = cc S + e: u - j comes from
// small terms only, so its rounding scales with the drag per step, not with
// |u| (a fixed fraction of u per step would be integrated by the slow Darcy
// relaxation).
//
// FIELD, FP32: w is held below 2^126, whose reciprocal is 0 and would leave the cell
// without any drag (from cc = 6.5e18 on, a porosity of 1e-9 at Da = 1e-6; the
// roots overflow at 1.8e19 and the step reports the divergence).  Held there, because the
// same bound on cc cost the one-step kernels 1.3 % (601 x 397 3.95 -> 4.00 us per step).
template <class V, bool FR, bool FIELD> __device__ __forceinline__ Vel<V> velocity(const Coll<Scalar<V>>& k, const Por<V>& p,
                                                                       const Sums<V>& s, V F) {
    Vel<V> m;
    m.dTl = op::add(s.n0, k.qhalf);
    m.dT = FR ? op::add(F, m.dTl) : m.dTl;
    const V by = op::mul(p.hb, m.dT);
    const V jx = op::add(s.ex, s.dx), jy = op::add(s.ey, s.dy);
    const V vy = op::add(jy, by);
    m.vm = op::root(op::fma(jx, jx, op::fma(vy, vy, op::tiny(V(0)))));
    const V e = op::fma(p.l1, m.vm, p.ec);
    m.S = op::add(op::root(op::add(V(Scalar<V>(0.25)), e)), V(Scalar<V>(0.5)));
    V w = op::fma(p.cc, m.S, e);
    if constexpr (FIELD) w = op::at_most(w, 4e37f);
    m.ngd = op::mul(w, op::minus_inverse(op::add(m.S, w)));
    m.dux = op::mul(jx, m.ngd);
    m.duy = op::fma(vy, m.ngd, by);
    m.ux = op::add(jx, m.dux);
    m.uy = op::add(jy, m.duy);
    return m;
}

// Eq. 22's quotient 1 / (l0 + sqrt(l0^2 + l1 |v|)).  1 + ngd is the same number, but
// its rounding is one of 1: where the drag is strong, little of it is right, or
// nothing (FP32: off by a percent or two at cc = 1e5, 0 or negative from 1e7 on).
template <class V> __device__ __forceinline__ V quotient(const Por<V>& p, const Vel<V>& m) {
    return op::inverse(op::add(p.cc, m.S));
}
// Whether the drag takes more than half of v (ngd < -1/2; a NaN may count as either), by the bits:
// off the FP64 unit.
__device__ __forceinline__ bool strong_drag(float ngd) { return __float_as_uint(ngd) > 0xBF000000u; }
__device__ __forceinline__ bool strong_drag(double ngd) { return (uint32_t)__double2hiint(ngd) >= 0xBFE00000u; }

// ---- collision -------------------------------------------------------------------------

// The increments of the flow populations from the combined moments: z and m0
// (energy), E (work of the force), p7, p8 (stress), and per direction the
// axis and diagonal parts of the momentum moments.
template <class V>
__device__ __forceinline__ void flow_out(const Coll<Scalar<V>>& k, V m0, V z, V E, bool with_E, V p7, V p8, V xa, V ya, V xd,
                                         V yd, V (&d)[9]) {
    V q0 = op::fma(k.a1, z, op::mul(k.a0, m0));
    V r1 = op::fma(k.b1, z, op::mul(k.b0, m0));
    V r5 = op::fma(k.c1, z, op::mul(k.c0, m0));
    if (with_E) {
        q0 = op::fma(k.a2, E, q0);
        r1 = op::fma(k.b2, E, r1);
        r5 = op::fma(k.c2, E, r5);
    }
    const V A = op::add(r1, p7), B = op::sub(r1, p7);
    const V G = op::add(r5, p8), H = op::sub(r5, p8);
    const V ds = op::add(xd, yd), dm = op::sub(xd, yd);
    d[0] = op::add(d[0], q0);
    d[1] = op::add(d[1], op::add(A, xa));
    d[3] = op::add(d[3], op::sub(A, xa));
    d[2] = op::add(d[2], op::add(B, ya));
    d[4] = op::add(d[4], op::sub(B, ya));
    d[5] = op::add(d[5], op::add(G, ds));
    d[7] = op::add(d[7], op::sub(G, ds));
    d[8] = op::add(d[8], op::add(H, dm));
    d[6] = op::add(d[6], op::sub(H, dm));
}

// Eq. 34-35 with Eq. 29-30 and the change of frame of the stored values: sh
// is the frame's change in units of k.w0, k.w1 (0 without frames); nf1 =
// n_1 - u_x T / sigma, nf2 likewise.
template <class V, bool FR>
__device__ __forceinline__ void heat_out(const Coll<Scalar<V>>& k, const Sums<V>& s, V nf1, V nf2, V sh, V (&h)[5]) {
    V U0 = V(k.q0), U1 = V(k.q1);
    if constexpr (FR) {
        U0 = op::fma(k.nw0, sh, U0);
        U1 = op::fma(k.nw1, sh, U1);
    }
    U0 = op::fma(k.t4, s.tt, op::fma(k.h4, h[0], U0));
    U1 = op::fma(k.t1, s.tt, op::fma(k.h1, h[0], U1));
    const V P = op::fma(k.z4, s.n4, U1), N = op::fma(k.nz4, s.n4, U1);
    const V g1 = op::mul(k.z1, nf1), g2 = op::mul(k.z2, nf2);
    h[0] = op::add(h[0], U0);
    h[1] = op::add(h[1], op::add(P, g1));
    h[3] = op::add(h[3], op::sub(P, g1));
    h[2] = op::add(h[2], op::add(N, g2));
    h[4] = op::add(h[4], op::sub(N, g2));
}

// |u| >= 1/2 or a non-finite value (Q = |u|^2 or vm, ngd give |u|).
__device__ __forceinline__ bool too_fast(const Vel<float>& m) { return !(op::fma(m.vm, m.ngd, m.vm) < 0.5f); }
__device__ __forceinline__ bool too_fast(const Vel<F2>& m) {
    const F2 u = op::fma(m.vm, m.ngd, m.vm);
    return !(u.v.x < 0.5f) || !(u.v.y < 0.5f);
}
// FP64: the exponent word decides, off the FP64 unit (a NaN is above).  Without its sign: under
// strong drag the sum may round to a negative number, of the size of |v| 2^-52.
__device__ __forceinline__ bool too_fast(const Vel<double>& m) {
    return (__double2hiint(op::fma(m.vm, m.ngd, m.vm)) & 0x7FFFFFFF) >= 0x3FE00000;
}

// Collision of a fluid node, in place on the pulled populations.
template <class V, bool FIELD, bool FR>
__device__ __forceinline__ void collide_fluid(const Coll<Scalar<V>>& k, const Por<V>& p, const Sums<V>& s, const Vel<V>& m,
                                              V sh, V (&d)[9], V (&h)[5]) {
    // with a porosity field the products carry 1 / phi, else the coefficients do
    const V uxp = FIELD ? op::mul(m.ux, p.iphi) : m.ux, uyp = FIELD ? op::mul(m.uy, p.iphi) : m.uy;
    const V P1 = op::mul(uxp, m.ux), P2 = op::mul(uyp, m.uy);
    const V T1 = op::mul(uxp, m.dux), T2 = op::mul(uyp, m.duy);
    const V Q = op::add(P1, P2), N7 = op::sub(P1, P2), C8 = op::mul(uxp, m.uy);
    const V E = op::add(T1, T2), D = op::sub(T1, T2);
    const V C = op::fma(uxp, m.duy, op::mul(uyp, m.dux));
    const V w = op::fms(Scalar<V>(4), s.b, s.a);
    const V z = FIELD ? op::sub(w, Q) : op::fma(k.niphi, Q, w);
    const V t7 = FIELD ? op::sub(s.m7, N7) : op::fma(k.niphi, N7, s.m7);
    const V t8 = FIELD ? op::sub(s.m8, C8) : op::fma(k.niphi, C8, s.m8);
    const V p7 = op::fma(k.k7, t7, op::mul(k.f7, D)), p8 = op::fma(k.k8, t8, op::mul(k.f8, C));
    const V m0 = op::add(d[0], op::add(s.a, s.b));
    const V t4 = op::fms(Scalar<V>(2), s.dx, s.ex), t6 = op::fms(Scalar<V>(2), s.dy, s.ey);
    const V xa = op::fma(k.s4a, t4, op::mul(V(2.0 / 3.0), m.dux)), ya = op::fma(k.s6a, t6, op::mul(V(2.0 / 3.0), m.duy));
    const V xd = op::fma(k.s4d, t4, op::mul(V(1.0 / 6.0), m.dux)), yd = op::fma(k.s6d, t6, op::mul(V(1.0 / 6.0), m.duy));
    flow_out(k, m0, z, E, true, p7, p8, xa, ya, xd, yd, d);
    const V nTs = op::fma(m.dT, k.nis, k.nTis);  // -T / sigma
    heat_out<V, FR>(k, s, op::fma(m.ux, nTs, s.n1), op::fma(m.uy, nTs, s.n2), sh, h);
}

// Collision of a wall node (u = 0) from its extrapolated populations: dux, duy
// = u - j, which the extrapolation takes over from the inner neighbour, and
// Fy = phi_b g beta (T_b - T0).
template <class V, bool FR>
__device__ __forceinline__ void collide_wall(const Coll<Scalar<V>>& k, V dux, V duy, V Fy, V sh, V (&d)[9], V (&h)[5]) {
    const Sums<V> s = sums_of(d, h);
    const V z = op::fms(Scalar<V>(4), s.b, s.a);
    const V m0 = op::add(d[0], op::add(s.a, s.b));
    const V t4 = op::fms(Scalar<V>(2), s.dx, s.ex), t6 = op::fms(Scalar<V>(2), s.dy, s.ey);
    // m_3, m_4 gain s (u - j) + (1 - s/2) F, in sixths: M = (m_3 part), N = (m_4 part)
    const V Mx = op::mul(k.s3, dux), Nx = op::mul(k.s4, dux);
    const V My = op::fma(k.f5, Fy, op::mul(k.s5, duy)), Ny = op::fma(k.f6, Fy, op::mul(k.s6, duy));
    const V xa = op::fma(k.s4a, t4, op::add(Mx, Nx)), ya = op::fma(k.s6a, t6, op::add(My, Ny));
    const V xd = op::fma(k.s4d, t4, op::fma(V(-0.5), Nx, Mx)), yd = op::fma(k.s6d, t6, op::fma(V(-0.5), Ny, My));
    flow_out(k, m0, z, z, false, op::mul(k.k7, s.m7), op::mul(k.k8, s.m8), xa, ya, xd, yd, d);
    heat_out<V, FR>(k, s, s.n1, s.n2, sh, h);
}

}  // namespace lbm
