// Reverse mode of one node of the fused step, for the discrete adjoint.
//
// The forward map of one node (pull, wall rule, collision; Sections 3-4), in
// the form of lbm_core.cuh, is differentiated by hand: given the adjoint of the
// node's post-collision populations (lambda for the flow, mu for the heat),
// these functions return the adjoint of the pulled populations that it read
// and of the porosity that it used.  Porosity enters through the per-cell Ergun
// drag (Eq. 4-5) and the equilibria (Eq. 14, 16, 19, 23).
//
// The rearranged collision has a short transpose.  It reads m_0, z, the stress
// and the energy-flux moments, j and n_0 only, the transpose needs the same eight
// sums of lambda as the forward step takes of f, and of the forward state it
// needs j and n_0 alone.  A wall node runs the collision with the moments z,
// m_0, t_7, t_8, t_4, t_6 of its inner neighbour (the extrapolated populations
// leave them unchanged), so its lambda adds to the neighbour's before the shared
// part of the transpose, and one pass through the velocity's derivative serves
// a fluid node and all the wall nodes that extrapolate from it.
// An interior node takes about 190 operations, 840 before that.
#pragma once

#include "lbm_node.cuh"

namespace lbm {

// Forward values at a fluid node; s holds j's four parts and n_0 only, and a, b
// next to a wall.
template <class V> struct Tape {
    Por<V> p;
    V r;  // (1 - phi) / phi
    Sums<V> s;
    Vel<V> m;
    V q;  // 1 + ngd
};

// u and 1 + ngd are taken from the quotient, to the rounding of each: seeds scale
// with them, and u's products enter the porosity's adjoint with 1 / phi^2, so what
// cancels in j + (u - j) would show there (nearly solid cells, FP32: gradients off by
// up to 3 %, now by 3e-5).
template <class V, bool FR>
__device__ __forceinline__ void tape_node(const Coll<Scalar<V>>& k, V phi, const Sums<V>& s, V F, Tape<V>& t) {
    t.p = por_of<V, true>(k, phi);
    t.r = op::mul(op::sub(V(1), phi), t.p.iphi);
    t.s = s;
    t.m = velocity<V, FR, true>(k, t.p, s, F);
    t.q = quotient(t.p, t.m);
    t.m.ux = op::mul(op::add(s.ex, s.dx), t.q);
    t.m.uy = op::mul(op::fma(t.p.hb, t.m.dT, op::add(s.ey, s.dy)), t.q);
}

// Seeds that the collision's transpose meets: of E, D, C (products of u and u -
// j) and of u - j, which only the node's own lambda gives, and what the wall
// rule adds to those of Q, N_7, C_8 (products of u), u, -T / sigma, T and 1 / phi.
template <class V> struct Seeds {
    V E, D, C, dux, duy;
    V Q, N7, C8, ux, uy, nT, dT, ip, dP;
};

template <class V>
__device__ __forceinline__ void own_seeds(const Coll<Scalar<V>>& k, V l0, const Sums<V>& l, Seeds<V>& b) {
    const V third = V(2.0 / 3.0), sixth = V(1.0 / 6.0);
    b.E = op::fma(k.c2, l.b, op::fma(k.b2, l.a, op::mul(k.a2, l0)));
    b.D = op::mul(k.f7, l.m7);
    b.C = op::mul(k.f8, l.m8);
    b.dux = op::fma(sixth, l.dx, op::mul(third, l.ex));
    b.duy = op::fma(sixth, l.dy, op::mul(third, l.ey));
}

// Adds a wall node's part to the seeds of its inner neighbour (tape t): l, l0,
// m0 are the sums and the rest populations of its lambda and mu.  Its flow
// populations are f_f - s(u_f) + c_P (dP_b - dP_f), its heat g_f + w~ (dT_b -
// dT_f) -+ T_f u_f / (2 sigma), its force phi_b g beta dT_b; an adiabatic wall
// (dirichlet = false) has dT_b = dT_f.  Returns the adjoint of phi_b.
template <class V>
__device__ __forceinline__ V wall_seeds(const Coll<V>& k, const Tape<V>& t, V phi_b, bool dirichlet, V dT_wall, V l0,
                                        V m0, const Sums<V>& l, Seeds<V>& b) {
    const V ux = t.m.ux, uy = t.m.uy;
    // sum_i lambda_i s_i = Q (-2/3 lambda_0 + (a + b) / 12) + N_7 m_7 / 4 + C_8 m_8 / 4 + u . (e / 3 + d / 12)
    b.Q = op::add(b.Q, op::fma(V(2.0 / 3.0), l0, op::mul(V(-1.0 / 12.0), op::add(l.a, l.b))));
    b.N7 = op::fma(V(-0.25), l.m7, b.N7);
    b.C8 = op::fma(V(-0.25), l.m8, b.C8);
    b.ux = op::sub(b.ux, op::fma(V(1.0 / 12.0), l.dx, op::mul(V(1.0 / 3.0), l.ex)));
    b.uy = op::sub(b.uy, op::fma(V(1.0 / 12.0), l.dy, op::mul(V(1.0 / 3.0), l.ey)));
    // pressure: dP_b - dP_f = (phi_b / phi_f - 1) (1/3 + dP_f)
    const V ddP = op::fma(V(-5.0 / 3.0), l0, op::fma(V(1.0 / 12.0), l.b, op::mul(V(1.0 / 3.0), l.a)));
    const V uip = op::mul(op::fma(ux, ux, op::mul(uy, uy)), t.p.iphi);
    const V P = op::add(V(1.0 / 3.0), op::fma(V(-0.4), uip, op::mul(V(0.6), op::add(t.s.a, t.s.b))));
    const V PddP = op::mul(P, ddP);
    b.ip = op::fma(phi_b, PddP, b.ip);
    b.dP = op::fma(op::fma(phi_b, t.p.iphi, V(-1)), ddP, b.dP);
    // momentum: M = s_3 (u - j), N = s_4 (u - j) (y: and the force), axis M + N, diagonal M - N / 2
    const V mx = op::add(l.ex, l.dx), nx = op::fma(V(-0.5), l.dx, l.ex);
    const V my = op::add(l.ey, l.dy), ny = op::fma(V(-0.5), l.dy, l.ey);
    b.dux = op::fma(k.s3, mx, op::fma(k.s4, nx, b.dux));
    b.duy = op::fma(k.s5, my, op::fma(k.s6, ny, b.duy));
    const V Fy = op::mul(k.gb, op::fma(k.f5, my, op::mul(k.f6, ny)));  // times phi_b dT_b
    // heat
    const V hnT = op::mul(V(0.5), op::fma(t.m.dT, k.nis, k.nTis));
    b.ux = op::fma(hnT, l.n1, b.ux);
    b.uy = op::fma(hnT, l.n2, b.uy);
    b.nT = op::fma(V(0.5), op::fma(ux, l.n1, op::mul(uy, l.n2)), b.nT);
    if (dirichlet) b.dT = op::sub(b.dT, op::fma(k.wt0, m0, op::mul(k.wt1, l.tt)));
    else b.dT = op::fma(phi_b, Fy, b.dT);
    return op::fma(t.p.iphi, PddP, op::mul(Fy, dirichlet ? dT_wall : t.m.dT));
}

// The transpose of a fluid node's step: l, m are lambda and mu (next to a wall
// those of the wall nodes included) and become the adjoint of the pulled
// populations; s their sums.  WALL: b holds wall nodes' parts.  Returns the
// adjoint of the porosity.
template <class V, bool WALL>
__device__ __forceinline__ V node_adjoint(const Coll<Scalar<V>>& k, const Tape<V>& t, const Seeds<V>& b, const Sums<V>& s,
                                          V (&l)[9], V (&m)[5]) {
    const Vel<V>& v = t.m;
    const V ip = t.p.iphi;
    // moments
    const V m0 = op::fma(k.c0, s.b, op::fma(k.b0, s.a, op::mul(k.a0, l[0])));
    const V z = op::fma(k.c1, s.b, op::fma(k.b1, s.a, op::mul(k.a1, l[0])));
    const V t7 = op::mul(k.k7, s.m7), t8 = op::mul(k.k8, s.m8);
    const V t4 = op::fma(k.s4d, s.dx, op::mul(k.s4a, s.ex)), t6 = op::fma(k.s6d, s.dy, op::mul(k.s6a, s.ey));
    // P_1 = Q + N_7, P_2 = Q - N_7 enter as 2 P_1 / u_x and so on
    V Q = -z, N7 = -t7, C8 = -t8, s18 = V(0);
    if constexpr (WALL) {
        Q = op::add(Q, op::fma(V(Scalar<V>(-0.4)), b.dP, b.Q));
        N7 = op::add(N7, b.N7);
        C8 = op::add(C8, b.C8);
        s18 = op::mul(V(Scalar<V>(0.6)), b.dP);
    }
    const V two = V(2), P1 = op::mul(two, op::add(Q, N7)), P2 = op::mul(two, op::sub(Q, N7));
    const V T1 = op::add(b.E, b.D), T2 = op::sub(b.E, b.D);
    const V Ax = op::fma(v.ux, P1, op::fma(v.uy, C8, op::fma(v.dux, T1, op::mul(v.duy, b.C))));
    const V Ay = op::fma(v.uy, P2, op::fma(v.ux, C8, op::fma(v.duy, T2, op::mul(v.dux, b.C))));
    const V Bx = op::fma(v.ux, T1, op::mul(v.uy, b.C)), By = op::fma(v.uy, T2, op::mul(v.ux, b.C));
    // the products are quadratic in (u, u - j): twice their sum
    V ipb = op::mul(V(Scalar<V>(0.5)),
                    op::fma(v.ux, Ax, op::fma(v.uy, Ay, op::fma(v.dux, Bx, op::mul(v.duy, By)))));
    // heat
    const V nT = op::fma(v.dT, k.nis, k.nTis);  // -T / sigma
    const V g1 = op::mul(k.z1, s.n1), g2 = op::mul(k.z2, s.n2), n4 = op::mul(k.z4, s.n4);
    V uxb = op::fma(ip, Ax, op::mul(nT, g1)), uyb = op::fma(ip, Ay, op::mul(nT, g2));
    V nTb = op::fma(v.ux, g1, op::mul(v.uy, g2));
    if constexpr (WALL) {
        ipb = op::add(ipb, b.ip);
        uxb = op::add(uxb, b.ux);
        uyb = op::add(uyb, b.uy);
        nTb = op::add(nTb, b.nT);
    }
    V dTb = op::mul(k.nis, nTb);
    if constexpr (WALL) dTb = op::add(dTb, b.dT);
    // velocity: u - j = -g v (y: + b), u = j + (u - j), b = hb dT, g = 1 - 1 / (cc + S)
    const V px = op::add(uxb, op::fma(ip, Bx, b.dux)), py = op::add(uyb, op::fma(ip, By, b.duy));
    const V by = op::mul(t.p.hb, v.dT);
    const V jx = op::add(t.s.ex, t.s.dx), vy = op::add(op::add(t.s.ey, t.s.dy), by);
    const V den = t.q;
    const V Sb = op::mul(op::fma(jx, px, op::mul(vy, py)), op::mul(-den, den));
    const V eb = op::mul(Sb, op::inverse(op::fma(two, v.S, V(-1))));  // e = l1 |v| + cc + cc^2 = S^2 - S
    const V ccb = op::fma(op::fma(two, t.p.cc, V(1)), eb, Sb), l1b = op::mul(eb, v.vm);
    const V rho = op::mul(op::mul(eb, t.p.l1), op::inverse(v.vm));  // |v| has derivative v / |v|, 0 at v = 0
    const V jxb = op::fma(jx, rho, op::fma(v.ngd, px, uxb));
    const V vyb = op::fma(vy, rho, op::mul(v.ngd, py));
    const V jyb = op::add(uyb, vyb), byb = op::add(py, vyb);
    dTb = op::fma(t.p.hb, byb, dTb);
    // porosity: cc = k.cc r^2, l1 = k.l1 r / phi, hb = k.hb phi, with r = 1 / phi - 1
    const V r2 = op::mul(two, t.r);
    const V ipt = op::fma(op::mul(k.cc, r2), ccb, op::fma(op::mul(k.l1, op::add(V(1), r2)), l1b, ipb));
    const V phib = op::fma(op::mul(k.hb, v.dT), byb, op::mul(op::mul(-ip, ip), ipt));
    // populations
    V a = op::sub(m0, z), bb = op::fma(V(4), z, m0);
    if constexpr (WALL) {
        a = op::add(a, s18);
        bb = op::add(bb, s18);
    }
    const V ex = op::sub(jxb, t4), ey = op::sub(jyb, t6);
    const V dx = op::fma(two, t4, jxb), dy = op::fma(two, t6, jyb);
    const V A = op::add(a, t7), B = op::sub(a, t7), G = op::add(bb, t8), H = op::sub(bb, t8);
    const V ds = op::add(dx, dy), dm = op::sub(dx, dy);
    l[0] = op::add(l[0], m0);
    l[1] = op::add(l[1], op::add(A, ex));
    l[3] = op::add(l[3], op::sub(A, ex));
    l[2] = op::add(l[2], op::add(B, ey));
    l[4] = op::add(l[4], op::sub(B, ey));
    l[5] = op::add(l[5], op::add(G, ds));
    l[7] = op::add(l[7], op::sub(G, ds));
    l[8] = op::add(l[8], op::add(H, dm));
    l[6] = op::add(l[6], op::sub(H, dm));
    const V U0 = op::fma(k.h1, s.tt, op::fma(k.h4, m[0], dTb));
    const V U1 = op::fma(k.t1, s.tt, op::fma(k.t4, m[0], dTb));
    const V Pp = op::add(U1, n4), Nn = op::sub(U1, n4);
    m[0] = op::add(m[0], U0);
    m[1] = op::add(m[1], op::add(Pp, g1));
    m[3] = op::add(m[3], op::sub(Pp, g1));
    m[2] = op::add(m[2], op::add(Nn, g2));
    m[4] = op::add(m[4], op::sub(Nn, g2));
    return phib;
}

}  // namespace lbm
