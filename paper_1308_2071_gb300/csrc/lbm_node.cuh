// One node, or two nodes, of the step: pull, wall rule (Section 4), collision,
// store; and the temperatures of the post-stream state that the Nusselt
// number reads.  FP32 and FP64 storage (Core<T>) run the collision of
// lbm_core.cuh, FP16 flow storage the direct form of lbm_device.cuh.
#pragma once

#include "lbm_core.cuh"

namespace lbm {

// ---- frames and pulled temperatures -------------------------------------------------

// The frame of node off in its unit (8-bit frames: the integer k, F = k fq;
// FP32 frames: F itself; none: 0).
template <class T>
__device__ __forceinline__ typename T::R core_frame(const Src<T>& src, const Geom& gm, int off) {
    using R = typename T::R;
    if constexpr (!Framed<T>::value)
        return R(0);
    else if constexpr (sizeof(typename FrameStore<T>::type) == 1)
        return in_plane(gm, off) ? R(frame_code<T>(src.t + off)) : R(0);
    else
        return in_plane(gm, off) ? Conv<typename FrameStore<T>::type, R, T::cg>::ld(src.t + off) : R(0);
}

// Framed storage: thermal values pulled into node off were stored in the
// frames of the nodes they came from; re-express them in this node's frame F
// (add w~_j (F(x - e_j) - F), j >= 1: differences of nearby frames are exact)
// and return F in its unit.
template <class T>
__device__ __forceinline__ typename T::R core_frame_in(const Coll<typename T::R>& k, const Src<T>& src,
                                                       const Geom& gm, int off, typename T::R (&h)[5]) {
    using R = typename T::R;
    if constexpr (!Framed<T>::value) {
        return R(0);
    } else {
        const R F = core_frame<T>(src, gm, off);
#pragma unroll
        for (int j = 1; j < 5; ++j)
            h[j] = op::fma(k.w1, op::sub(core_frame<T>(src, gm, off - ey9(j) * gm.pitch - ex9(j)), F), h[j]);
        return F;
    }
}

// The same for the node pair off0, off0 + 1 (x0 even): the pair's own frames
// and those of the rows above and below come as pairs.
template <class T>
__device__ __forceinline__ void core_frame_in_x2(const Coll<typename T::R>& k, const Src<T>& src, const Geom& gm,
                                                 int off0, typename T::R (&h0)[5], typename T::R (&h1)[5],
                                                 typename T::R& F0, typename T::R& F1) {
    using R = typename T::R;
    F0 = F1 = R(0);
    if constexpr (Framed<T>::value) {
        R n0 = R(0), n1 = R(0), s0 = R(0), s1 = R(0);
        auto pair = [&](int delta, R& a, R& b) {
            if (!in_plane(gm, off0 + delta, 2)) return;
            if constexpr (sizeof(typename FrameStore<T>::type) == 1) {
                const char2 v = frame_pair_code<T>(at(src.t, delta, off0));
                a = R((int)(signed char)v.x);
                b = R((int)(signed char)v.y);
            } else {
                const auto v = Conv2<typename FrameStore<T>::type, R, T::cg>::ld(at(src.t, delta, off0));
                a = v.x;
                b = v.y;
            }
        };
        pair(0, F0, F1);
        pair(-gm.pitch, s0, s1);  // j = 2: y - 1
        pair(gm.pitch, n0, n1);  // j = 4: y + 1
        auto one = [&](int delta) {
            if (!in_plane(gm, off0 + delta)) return R(0);
            if constexpr (sizeof(typename FrameStore<T>::type) == 1) return R(frame_code<T>(at(src.t, delta, off0)));
            else return Conv<typename FrameStore<T>::type, R, T::cg>::ld(at(src.t, delta, off0));
        };
        const R w = one(-1), e = one(2);
        const R dF = op::sub(F1, F0);
        h0[1] = op::fma(k.w1, op::sub(w, F0), h0[1]);
        h1[1] = op::fma(k.w1, -dF, h1[1]);
        h0[2] = op::fma(k.w1, op::sub(s0, F0), h0[2]);
        h1[2] = op::fma(k.w1, op::sub(s1, F1), h1[2]);
        h0[3] = op::fma(k.w1, dF, h0[3]);
        h1[3] = op::fma(k.w1, op::sub(e, F1), h1[3]);
        h0[4] = op::fma(k.w1, op::sub(n0, F0), h0[4]);
        h1[4] = op::fma(k.w1, op::sub(n1, F1), h1[4]);
    }
}

// The frame a node takes for the temperature deviation dT: its value in the
// frames' unit (next) and stored form (code); returns its change from the
// frame F.  8-bit frames: k = round(dT / fq) by adding 1.5 * 2^23 (the product
// is exact, so this rounds once, to nearest even), clamped to 8 bits; a NaN or
// an overflowing value saturates (the divergence flag reports it).
template <class T>
__device__ __forceinline__ typename T::R frame_next(const Coll<typename T::R>& k, typename T::R dT, typename T::R F,
                                                    typename T::R& next, typename FrameStore<T>::type& code) {
    using R = typename T::R;
    if constexpr (!Framed<T>::value) {
        return next = R(0);
    } else if constexpr (sizeof(typename FrameStore<T>::type) == 1) {
        constexpr float big = 12582912.f;
        const float t = fminf(fmaxf(op::fma(dT, k.ifu, big), big - 128.f), big + 127.f);
        code = (typename FrameStore<T>::type)(__float_as_int(t) & 0xff);
        next = op::sub(t, big);
        return op::sub(next, F);
    } else {
        next = code = dT;
        return op::sub(dT, F);
    }
}
// The same for two nodes.
template <class T>
__device__ __forceinline__ F2 frame_next(const Coll<float>& k, F2 dT, F2 F, F2& next,
                                         typename FrameStore<T>::type& code0, typename FrameStore<T>::type& code1) {
    if constexpr (sizeof(typename FrameStore<T>::type) == 1) {
        constexpr float big = 12582912.f;
        const F2 u = op::fma(dT, k.ifu, big);
        const F2 t(fminf(fmaxf(u.v.x, big - 128.f), big + 127.f), fminf(fmaxf(u.v.y, big - 128.f), big + 127.f));
        code0 = (typename FrameStore<T>::type)(__float_as_int(t.v.x) & 0xff);
        code1 = (typename FrameStore<T>::type)(__float_as_int(t.v.y) & 0xff);
        next = op::add(t, -big);
    } else {
        next = dT;
        code0 = dT.v.x;
        code1 = dT.v.y;
    }
    return op::sub(next, F);
}

// Thermal values pulled into node off (framed: in its frame F, in its unit).
template <class T>
__device__ __forceinline__ typename T::R pull_heat(const CoefOf<T>& c, const Src<T>& src, const Geom& gm,
                                                   int off, typename T::R& F) {
    using R = typename T::R;
    R h[5];
#pragma unroll
    for (int j = 0; j < 5; ++j) {
        const int o = off - ey9(j) * gm.pitch - ex9(j);
        h[j] = in_plane(gm, o) ? Conv<typename T::SG, R, T::cg>::ld(src.g + j * gm.plane + o) : R(0);
    }
    if constexpr (Core<T>::value) {
        F = op::mul(core_frame_in<T>(c.k, src, gm, off, h), c.k.fu);
        return heat(h);
    } else {
        F = frame_in<T>(c, src, gm, off, h);
        return h[0] + h[1] + h[2] + h[3] + h[4];
    }
}

// ---- wall rule ----------------------------------------------------------------------------

// Inward normal of a node: (0, 0) for fluid nodes, the diagonal at corners.
struct Normal {
    int dx, dy;
};
__device__ __forceinline__ Normal normal_of(const Geom& gm, int x, int y) {
    Normal n;
    n.dx = (x == 0) ? 1 : (x == gm.nx - 1 ? -1 : 0);
    n.dy = (y == 0) ? 1 : (y == gm.ny - 1 ? -1 : 0);
    return n;
}

// Non-equilibrium extrapolation (Section 4, ref. [43]) at wall node (x, y)
// with inward normal nr: reads the pulled populations of the inner neighbour
// x_f = x + nr (and of x + 2 nr for the second-order adiabatic variant),
// writes the wall node's populations into d, h and returns the imposed
// macroscopic values (u = 0, p_b = p_f, T_b; force phi_b G(T_b) j).  FP16 flow
// storage; core_wall below is the same rule for FP32 and FP64.
template <class T, bool FIELD>
__device__ __forceinline__ Macro<typename T::R> wall_node(const Direct& c, const Geom& gm,
                                                          const Src<T>& src, const typename T::P* phi_field,
                                                          int x, int y, Normal nr,
                                                          const Drag<typename T::R>& drb,
                                                          typename T::R (&d)[9], typename T::R (&h)[5]) {
    using R = typename T::R;
    const int offf = (y + nr.dy) * gm.pitch + (x + nr.dx);
    R df[9], hf[5];
    pull<T>(src, gm, offf, df, hf);
    // frames of the inner neighbour and of this wall node
    const R Ff = frame_in<T>(c, src, gm, offf, hf);
    const R Fb = in_plane(gm, y * gm.pitch + x) ? frame_ld<T>(c, src.t + y * gm.pitch + x) : R(0);
    const Drag<R> drf = drag_at<R, FIELD, typename T::P>(c, gm, phi_field, offf);
    const Macro<R> mf = fluid_macros<R>(c, drf, df, hf, Ff);

    Macro<R> mb;
    mb.ux = R(0);
    mb.uy = R(0);
    mb.umag = R(0);
    // p_b = p_f:  P_b = phi_b p_f, P = rho0 c_s^2 + dP
    if constexpr (FIELD) {
        mb.dP = (drb.phi * drf.iphi) * (R(1.0 / 3.0) + mf.dP) - R(1.0 / 3.0);
    } else {
        mb.dP = mf.dP;
    }
    const bool dirichlet = (gm.thermal_bc == 1) || (nr.dx != 0);
    // the wall temperature relative to this node's frame, from differences of nearby frames
    mb.F = Fb;
    if (dirichlet) {
        mb.dTl = ((gm.thermal_bc == 1) ? c.dTc : (x == 0 ? c.dTh : c.dTc)) - Fb;
    } else if (gm.adi_order == 2) {
        const int offff = (y + 2 * nr.dy) * gm.pitch + (x + 2 * nr.dx);
        R Fff;
        const R dTlff = pull_heat<T>(c, src, gm, offff, Fff) + c.qhalf;
        mb.dTl = (R(4) * ((Ff - Fb) + mf.dTl) - ((Fff - Fb) + dTlff)) * R(1.0 / 3.0);
    } else {
        mb.dTl = (Ff - Fb) + mf.dTl;
    }
    mb.dT = Fb + mb.dTl;
    mb.Fx = R(0);
    mb.Fy = drb.phi * c.gbeta * mb.dT;

    // f_b = f_eq(P_b, 0) + f_f - f_eq(P_f, u_f) (Eq. 13-14 as deviations):
    // f_eq,i - w_i rho0 = 3 w_i dP + s_i(u) (i >= 1), -(5/3) dP + s_0(u) (i = 0)
    const R ddP = mb.dP - mf.dP;
    const R ux = mf.ux, uy = mf.uy;
    const R uu = ux * ux + uy * uy;
    const R ip = drf.iphi;
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        const R eu = R(ex9(i)) * ux + R(ey9(i)) * uy;
        const R si = R(w9(i)) * (R(3) * eu + R(4.5) * eu * eu * ip - R(1.5) * uu * ip);
        const R cP = (i == 0) ? R(-5.0 / 3.0) : R(3.0 * w9(i));
        d[i] = df[i] - si + cP * ddP;
    }
    // g_b = g_eq(T_b, 0) + g_f - g_eq(T_f, u_f) (Eq. 37, first occurrence), in this node's
    // frame: w~ (T_b - T_f) + w~ (F_f - F_b) = w~ (dTl_b - dTl_f)
    const R Tf = c.T0 + mf.dT;
    const R ddT = mb.dTl - mf.dTl;
    const R adv = Tf * c.inv_sigma * c.inv_csT2 * c.wt1;
    const R sh0 = c.wt0 * ddT;
    const R sh1 = c.wt1 * ddT;
    h[0] = hf[0] + sh0;
    h[1] = hf[1] + sh1 - adv * ux;
    h[2] = hf[2] + sh1 - adv * uy;
    h[3] = hf[3] + sh1 + adv * ux;
    h[4] = hf[4] + sh1 + adv * uy;
    return mb;
}

// The same rule from values in registers (FP32 and FP64 storage): d, h hold the
// inner neighbour's pulled populations (porosity phi_f, sums s, velocity v,
// frame Ff in its unit) and become the wall node's (porosity phi_b, its own
// frame).  dTl: the imposed temperature T_b - T0 relative to the wall node's
// frame.  p_b - p_f enters through (phi_b - phi_f) / phi_f, exact where the
// porosity is uniform.  Returns dP_b; u_b - j_b equals u_f - j_f.
template <class R, bool FIELD>
__device__ __forceinline__ R core_wall(const Coll<R>& k, const Por<R>& pf, R phi_f, R phi_b, const Sums<R>& s,
                                       const Vel<R>& v, R dTl, R (&d)[9], R (&h)[5]) {
    const R uu = op::fma(v.ux, v.ux, op::mul(v.uy, v.uy));
    const R uip = op::mul(uu, pf.iphi);
    const R dPf = op::fma(R(-0.4), uip, op::mul(R(0.6), op::add(s.a, s.b)));
    R ddP = R(0);
    if constexpr (FIELD) ddP = op::mul(op::mul(op::sub(phi_b, phi_f), pf.iphi), op::add(R(1.0 / 3.0), dPf));
    // f_b = f_eq(P_b, 0) + f_f - f_eq(P_f, u_f) (Eq. 13-14 as deviations):
    // f_eq,i - w_i rho0 = 3 w_i dP + s_i(u) (i >= 1), -(5/3) dP + s_0(u) (i = 0)
    const R base = op::mul(R(-1.5), uip), q = op::mul(R(4.5), pf.iphi);
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        const R eu = op::add(ex9(i) == 0 ? R(0) : ex9(i) > 0 ? v.ux : -v.ux,
                             ey9(i) == 0 ? R(0) : ey9(i) > 0 ? v.uy : -v.uy);
        const R si = op::mul(R(w9(i)), op::fma(R(3), eu, op::fma(q, op::mul(eu, eu), base)));
        d[i] = op::sub(d[i], si);
        if constexpr (FIELD) d[i] = op::fma(i == 0 ? R(-5.0 / 3.0) : R(3.0 * w9(i)), ddP, d[i]);
    }
    // g_b = g_eq(T_b, 0) + g_f - g_eq(T_f, u_f) (Eq. 37, first occurrence; w~_1 /
    // c_sT^2 = 1/2), relative to the frames: w~ (T_b - T_f) + w~ (F_f - F_b) = w~ (dTl_b - dTl_f)
    const R ddT = op::sub(dTl, v.dTl);
    const R adv = op::mul(R(0.5), op::fma(v.dT, k.is, k.Tis));
    const R s1 = op::mul(k.wt1, ddT);
    h[0] = op::fma(k.wt0, ddT, h[0]);
    h[1] = op::fma(-adv, v.ux, op::add(h[1], s1));
    h[2] = op::fma(-adv, v.uy, op::add(h[2], s1));
    h[3] = op::fma(adv, v.ux, op::add(h[3], s1));
    h[4] = op::fma(adv, v.uy, op::add(h[4], s1));
    return op::add(dPf, ddP);
}

// Post-stream state of node (x, y) (pull + wall rule): a fluid node's own
// pulled populations, or, on a wall, those of its inner neighbour turned into
// the wall node's (the same loads and macroscopic values, from one node
// further in).
template <class R> struct Post {
    bool wall;
    Por<R> por;   // of the node the populations were pulled into
    Sums<R> s;
    Vel<R> v;
    R F;          // this node's frame in its unit
    R dTl, dT;    // this node's T - T0 - F and T - T0
    R dP, Fy;     // wall nodes: phi p - rho0 c_s^2 and the force
};
// Where core_post reads a lattice B_n: from its buffer, by node offset.
template <class T> struct BufferSource {
    using R = typename T::R;
    const Coef<R>& c;
    const Geom& gm;
    const Src<T>& src;
    // the populations pulled into node (x, y), the thermal ones in its frame, which is returned
    __device__ __forceinline__ R pulled(int x, int y, R (&d)[9], R (&h)[5]) const {
        const int off = y * gm.pitch + x;
        pull<T>(src, gm, off, d, h);
        return core_frame_in<T>(c.k, src, gm, off, h);
    }
    __device__ __forceinline__ R frame(int x, int y) const { return core_frame<T>(src, gm, y * gm.pitch + x); }
    // T - T0 - F of node (x, y) without the source half-step, and F
    __device__ __forceinline__ R heat_at(int x, int y, R& F) const {
        return pull_heat<T>(c, src, gm, y * gm.pitch + x, F);
    }
};
template <class T, bool FIELD, class Source>
__device__ __forceinline__ Post<typename T::R> core_post(const Coll<typename T::R>& k, const Geom& gm,
                                                         const Source& from, const typename T::P* phi, int x, int y,
                                                         typename T::R (&d)[9], typename T::R (&h)[5]) {
    using R = typename T::R;
    constexpr bool FR = Framed<T>::value;
    const Normal nr = normal_of(gm, x, y);
    const int xf = x + nr.dx, yf = y + nr.dy;
    const int off = y * gm.pitch + x, offf = yf * gm.pitch + xf;
    Post<R> p;
    p.wall = nr.dx != 0 || nr.dy != 0;
    const R Ff = from.pulled(xf, yf, d, h);
    const R phi_f = FIELD ? (in_plane(gm, offf) ? Conv<typename T::P, R>::ld(phi + offf) : R(1)) : R(0);
    p.por = por_of<R, FIELD>(k, phi_f);
    p.s = sums_of(d, h);
    p.v = velocity<R, FR, FIELD>(k, p.por, p.s, op::mul(Ff, k.fu));
    p.F = Ff;
    p.dTl = p.v.dTl;
    p.dT = p.v.dT;
    p.dP = p.Fy = R(0);
    if (p.wall) {
        const R phi_b = FIELD ? (in_plane(gm, off) ? Conv<typename T::P, R>::ld(phi + off) : R(1)) : R(0);
        p.F = from.frame(x, y);
        const R Fb = op::mul(p.F, k.fu), dF = op::mul(op::sub(Ff, p.F), k.fu);
        if (gm.thermal_bc == 1 || nr.dx != 0) {
            p.dTl = op::sub(gm.thermal_bc == 0 && x == 0 ? k.dTh : k.dTc, Fb);
        } else {
            p.dTl = op::add(dF, p.v.dTl);
            if (gm.adi_order == 2) {
                R Fff;
                const R l2 = from.heat_at(xf + nr.dx, yf + nr.dy, Fff);
                const R t2 = op::add(op::sub(Fff, Fb), op::add(l2, k.qhalf));
                p.dTl = op::mul(op::fma(R(4), p.dTl, -t2), R(1.0 / 3.0));
            }
        }
        p.dT = FR ? op::add(Fb, p.dTl) : p.dTl;
        p.dP = core_wall<R, FIELD>(k, p.por, phi_f, phi_b, p.s, p.v, p.dTl, d, h);
        p.Fy = op::mul(FIELD ? op::mul(phi_b, k.gb) : op::mul(R(2), k.hb), p.dT);
    }
    return p;
}

// Collides a node's post-stream populations in place; sh: the change of its frame.
template <class T, bool FIELD>
__device__ __forceinline__ void core_collide(const Coll<typename T::R>& k, const Post<typename T::R>& p,
                                             typename T::R sh, typename T::R (&d)[9], typename T::R (&h)[5]) {
    using R = typename T::R;
    if (p.wall)
        collide_wall<R, Framed<T>::value>(k, p.v.dux, p.v.duy, p.Fy, sh, d, h);
    else
        collide_fluid<R, FIELD, Framed<T>::value>(k, p.por, p.s, p.v, sh, d, h);
}

// Post-stream state of node (x, y) (pull + wall rule) and its macroscopic values.
template <class T, bool FIELD>
__device__ __forceinline__ Macro<typename T::R> node_state(const CoefOf<T>& c, const Geom& gm,
                                                           const Src<T>& src, const typename T::P* phi_field,
                                                           int x, int y, Drag<typename T::R>& dr,
                                                           typename T::R (&d)[9], typename T::R (&h)[5]) {
    using R = typename T::R;
    const int off = y * gm.pitch + x;
    if constexpr (Core<T>::value) {
        dr.phi = c.phi;
        if constexpr (FIELD) dr.phi = in_plane(gm, off) ? Conv<typename T::P, R>::ld(phi_field + off) : R(1);
        dr.iphi = R(1) / dr.phi;
        const Post<R> p = core_post<T, FIELD>(c.k, gm, BufferSource<T>{c, gm, src}, phi_field, x, y, d, h);
        Macro<R> m;
        // u and |u| as the step forms them, j + (u - j) and |v| (1 + ngd), or, where the drag takes
        // more than half of v and they cancel, from the quotient
        const R z = R(0), uu = op::fma(p.v.ux, p.v.ux, op::mul(p.v.uy, p.v.uy));
        m.ux = p.v.ux;
        m.uy = p.v.uy;
        m.umag = op::fma(p.v.vm, p.v.ngd, p.v.vm);
        if (strong_drag(p.v.ngd)) {
            const R q = quotient(p.por, p.v);
            m.ux = op::mul(op::add(p.s.ex, p.s.dx), q);
            m.uy = op::mul(op::fma(p.por.hb, p.v.dT, op::add(p.s.ey, p.s.dy)), q);
            m.umag = op::mul(p.v.vm, q);
        }
        if (p.wall) m.ux = m.uy = z;
        if (m.ux == z && m.uy == z) m.umag = z;  // at rest too: |v| has a floor (see tiny)
        m.dP = p.wall ? p.dP : op::fma(R(-0.4), op::mul(uu, p.por.iphi), op::mul(R(0.6), op::add(p.s.a, p.s.b)));
        m.dT = p.dT;
        m.dTl = p.dTl;
        m.F = op::mul(p.F, c.k.fu);
        return m;
    } else {
        dr = drag_at<R, FIELD, typename T::P>(c, gm, phi_field, off);
        const Normal nr = normal_of(gm, x, y);
        if (nr.dx == 0 && nr.dy == 0) {
            pull<T>(src, gm, off, d, h);
            const R F = frame_in<T>(c, src, gm, off, h);
            return fluid_macros<R>(c, dr, d, h, F);
        }
        return wall_node<T, FIELD>(c, gm, src, phi_field, x, y, nr, dr, d, h);
    }
}

// The populations of the post-stream state alone; returns the frame of the thermal
// ones.  A fluid node needs no macroscopic values for them (FP64 at 1024^2: 75 of 174
// us of a state read).
template <class T, bool FIELD>
__device__ __forceinline__ typename T::R node_populations(const CoefOf<T>& c, const Geom& gm,
                                                          const Src<T>& src, const typename T::P* phi_field, int x,
                                                          int y, typename T::R (&d)[9], typename T::R (&h)[5]) {
    const Normal nr = normal_of(gm, x, y);
    if (nr.dx == 0 && nr.dy == 0) {
        const int off = y * gm.pitch + x;
        pull<T>(src, gm, off, d, h);
        if constexpr (Core<T>::value) return op::mul(core_frame_in<T>(c.k, src, gm, off, h), c.k.fu);
        else return frame_in<T>(c, src, gm, off, h);
    }
    Drag<typename T::R> dr;
    return node_state<T, FIELD>(c, gm, src, phi_field, x, y, dr, d, h).F;
}

// FP16 flow storage: re-expresses the collided thermal values, relative to the
// frame mc.F they were computed in, in the node's new frame (T - T0 in the
// frame's storage type) and stores that frame.
template <class T>
__device__ __forceinline__ void frame_out(const Direct& c, const Geom& gm, const Dst<T>& dst, int off,
                                          const Macro<float>& mc, float (&h)[5]) {
    int8_t code;
    const float Fn = frame_make(c, mc.dT, code);  // F + dTl as the frame stores it: the new frame
    const float shift = Fn - mc.F;                 // exact: both are frame values
    h[0] -= c.wt0 * shift;
#pragma unroll
    for (int j = 1; j < 5; ++j) h[j] -= c.wt1 * shift;
    if (in_plane(gm, off)) dst.t[off] = code;
}

// ---- wall-column temperatures -------------------------------------------------------

// The Nusselt number (Eq. 38) reads T at the five node columns next to each
// vertical wall.  An observing step stores T - T0 of those nodes of the
// post-stream state as it computes them: obs[kObsCols y + k] holds node
// x = k (k < 5) and node x = nx - 1 - (k - 5) (k >= 5), in FP64, the value
// node_dT reports for a node off the walls (framed storage: frame and local
// part added in FP64).  A node of a narrow lattice may fill two slots.
constexpr int kObsCols = 10;

__device__ __forceinline__ void obs_put(const Geom& gm, double* obs, int x, int y, double v) {
    if (x < 5) obs[kObsCols * y + x] = v;
    if (x >= gm.nx - 5) obs[kObsCols * y + 5 + (gm.nx - 1 - x)] = v;
}

// One fluid node of the step (FP32 and FP64 storage).
template <class T, bool FIELD, bool OBS>
__device__ __forceinline__ void update_fluid(const Coef<typename T::R>& c, const Geom& gm, const Src<T>& src,
                                             const Dst<T>& dst, const typename T::P* __restrict__ phi, int x, int y,
                                             int* status, double* obs) {
    using R = typename T::R;
    constexpr bool FR = Framed<T>::value;
    const Coll<R>& k = c.k;
    const int off = y * gm.pitch + x;
    R d[9], h[5];
    pull<T>(src, gm, off, d, h);
    const R F = core_frame_in<T>(k, src, gm, off, h);
    const R phi_n = FIELD ? (in_plane(gm, off) ? Conv<typename T::P, R>::ld(phi + off) : R(1)) : R(0);
    const Por<R> p = por_of<R, FIELD>(k, phi_n);
    const Sums<R> s = sums_of(d, h);
    const Vel<R> v = velocity<R, FR, FIELD>(k, p, s, op::mul(F, k.fu));
    if (too_fast(v)) atomicOr(status, 1);  // also catches NaN
    typename FrameStore<T>::type code;
    R next;
    const R shift = frame_next<T>(k, v.dT, F, next, code);
    collide_fluid<R, FIELD, FR>(k, p, s, v, shift, d, h);
    if (in_plane(gm, off)) {
        if constexpr (FR) dst.t[off] = code;
#pragma unroll
        for (int i = 0; i < 9; ++i) Conv<typename T::SF, R, T::cg>::st(dst.f + i * gm.plane + off, d[i]);
#pragma unroll
        for (int j = 0; j < 5; ++j) Conv<typename T::SG, R, T::cg>::st(dst.g + j * gm.plane + off, h[j]);
    }
    if constexpr (OBS) obs_put(gm, obs, x, y, FR ? (double)op::mul(F, k.fu) + (double)v.dTl : (double)v.dT);
}

// One node of the step: pull (or wall rule), collide, store; OBS: also the
// node's temperature into obs when it lies in a wall column.  That store
// comes after all arithmetic: a branch between the macroscopic values and
// the collision would change where the compiler fuses multiply-adds, and
// with it the rounding of the lattice.
template <class T, bool FIELD, bool OBS = false>
__device__ __forceinline__ void update_node(const CoefOf<T>& c, const Geom& gm, const Src<T>& src,
                                            const Dst<T>& dst, const typename T::P* phi, int x, int y,
                                            int* status, double* obs = nullptr) {
    using R = typename T::R;
    R d[9], h[5];
    if constexpr (Core<T>::value) {
        const int off = y * gm.pitch + x;
        const Post<R> p = core_post<T, FIELD>(c.k, gm, BufferSource<T>{c, gm, src}, phi, x, y, d, h);
        if (!p.wall && too_fast(p.v)) atomicOr(status, 1);  // also catches NaN
        typename FrameStore<T>::type code;
        R next;
        const R sh = frame_next<T>(c.k, p.dT, p.F, next, code);
        core_collide<T, FIELD>(c.k, p, sh, d, h);
        if (in_plane(gm, off)) {
            if constexpr (Framed<T>::value) dst.t[off] = code;
#pragma unroll
            for (int i = 0; i < 9; ++i) Conv<typename T::SF, R, T::cg>::st(dst.f + i * gm.plane + off, d[i]);
#pragma unroll
            for (int j = 0; j < 5; ++j) Conv<typename T::SG, R, T::cg>::st(dst.g + j * gm.plane + off, h[j]);
        }
        if constexpr (OBS)
            obs_put(gm, obs, x, y, Framed<T>::value ? (double)op::mul(p.F, c.k.fu) + (double)p.dTl : (double)p.dT);
    } else {
        Drag<R> dr;
        const Macro<R> mc = node_state<T, FIELD>(c, gm, src, phi, x, y, dr, d, h);
        if (!(mc.umag < R(0.5))) atomicOr(status, 1);  // also catches NaN
        collide<R>(c, dr.iphi, mc, d, h);
        dither_to_half(d);
        const int off = y * gm.pitch + x;
        frame_out<T>(c, gm, dst, off, mc, h);
        if (in_plane(gm, off)) {
#pragma unroll
            for (int i = 0; i < 9; ++i) Conv<typename T::SF, R, T::cg>::st(dst.f + i * gm.plane + off, d[i]);
#pragma unroll
            for (int j = 0; j < 5; ++j) Conv<typename T::SG, R, T::cg>::st(dst.g + j * gm.plane + off, h[j]);
        }
        if constexpr (OBS) obs_put(gm, obs, x, y, (double)mc.F + (double)mc.dTl);
    }
}

// Two fluid nodes from their pulled values in one pass of F2 arithmetic (FP16 flow
// storage): about half the arithmetic instructions of two nodes.  F0, F1: the
// frames that the pulled thermal values b0, b1 are relative to (frame_in).
// VEC: the nodes are x-neighbours off1 = off0 + 1 with x0 even, stored as
// pairs.
template <class T, bool OBS = false, bool VEC = false>
__device__ __forceinline__ void collide_fluid_pair_x2(const Direct& c, const Geom& gm, const Dst<T>& dst,
                                                      const float (&a0)[9], const float (&b0)[5],
                                                      const float (&a1)[9], const float (&b1)[5],
                                                      const Drag<float>& r0, const Drag<float>& r1, int off0,
                                                      int off1, int* status, int x0, int y0, int x1, int y1,
                                                      double* obs, float F0, float F1) {
    Drag<F2> dr;
    dr.phi = F2(r0.phi, r1.phi);
    dr.iphi = F2(r0.iphi, r1.iphi);
    dr.c_lin = F2(r0.c_lin, r1.c_lin);
    dr.c_quad = F2(r0.c_quad, r1.c_quad);
    F2 d[9], h[5];
#pragma unroll
    for (int i = 0; i < 9; ++i) d[i] = F2(a0[i], a1[i]);
#pragma unroll
    for (int j = 0; j < 5; ++j) h[j] = F2(b0[j], b1[j]);
    const Macro<F2> m = fluid_macros<F2>(c, dr, d, h, F2(F0, F1));
    if (!(m.umag.v.x < 0.5f) || !(m.umag.v.y < 0.5f)) atomicOr(status, 1);
    collide<F2>(c, dr.iphi, m, d, h);
    {
        float v0[9], v1[9];
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            v0[i] = d[i].v.x;
            v1[i] = d[i].v.y;
        }
        dither_to_half(v0);
        dither_to_half(v1);
#pragma unroll
        for (int i = 0; i < 9; ++i) d[i] = F2(v0[i], v1[i]);
    }
    int8_t k0, k1;
    const float s0 = frame_make(c, m.dT.v.x, k0) - m.F.v.x;  // exact: frame values
    const float s1 = frame_make(c, m.dT.v.y, k1) - m.F.v.y;
    const F2 sh(s0, s1);
    h[0] = h[0] - c.wt0 * sh;
#pragma unroll
    for (int j = 1; j < 5; ++j) h[j] = h[j] - c.wt1 * sh;
    if constexpr (VEC) {
        if (in_plane(gm, off0, 2)) frame_st2<T>(at(dst.t, 0, off0), k0, k1);
    } else {
        if (in_plane(gm, off0)) dst.t[off0] = k0;
        if (in_plane(gm, off1)) dst.t[off1] = k1;
    }
    if constexpr (VEC) {
        if (in_plane(gm, off0, 2)) {
#pragma unroll
            for (int i = 0; i < 9; ++i)
                Conv2<typename T::SF, float, T::cg>::st(at(dst.f, i * gm.plane, off0), d[i].v.x, d[i].v.y);
#pragma unroll
            for (int j = 0; j < 5; ++j)
                Conv2<typename T::SG, float, T::cg>::st(at(dst.g, j * gm.plane, off0), h[j].v.x, h[j].v.y);
        }
    } else {
        if (in_plane(gm, off0)) {
#pragma unroll
            for (int i = 0; i < 9; ++i) Conv<typename T::SF, float, T::cg>::st(dst.f + i * gm.plane + off0, d[i].v.x);
#pragma unroll
            for (int j = 0; j < 5; ++j) Conv<typename T::SG, float, T::cg>::st(dst.g + j * gm.plane + off0, h[j].v.x);
        }
        if (in_plane(gm, off1)) {
#pragma unroll
            for (int i = 0; i < 9; ++i) Conv<typename T::SF, float, T::cg>::st(dst.f + i * gm.plane + off1, d[i].v.y);
#pragma unroll
            for (int j = 0; j < 5; ++j) Conv<typename T::SG, float, T::cg>::st(dst.g + j * gm.plane + off1, h[j].v.y);
        }
    }
    if constexpr (OBS) {
        // lane-wise IEEE sums: the same values as the scalar path
        obs_put(gm, obs, x0, y0, (double)m.F.v.x + (double)m.dTl.v.x);
        obs_put(gm, obs, x1, y1, (double)m.F.v.y + (double)m.dTl.v.y);
    }
}

template <class T, bool FIELD, bool OBS = false>
__device__ __forceinline__ void update_fluid_pair_x2(const Direct& c, const Geom& gm, const Src<T>& src,
                                                     const Dst<T>& dst, const typename T::P* phi, int x0, int y0,
                                                     int x1, int y1, int* status, double* obs = nullptr) {
    const int off0 = y0 * gm.pitch + x0, off1 = y1 * gm.pitch + x1;
    float a0[9], b0[5], a1[9], b1[5];
    pull<T>(src, gm, off0, a0, b0);
    pull<T>(src, gm, off1, a1, b1);
    const float F0 = frame_in<T>(c, src, gm, off0, b0);
    const float F1 = frame_in<T>(c, src, gm, off1, b1);
    const Drag<float> r0 = drag_at<float, FIELD, typename T::P>(c, gm, phi, off0);
    const Drag<float> r1 = drag_at<float, FIELD, typename T::P>(c, gm, phi, off1);
    collide_fluid_pair_x2<T, OBS>(c, gm, dst, a0, b0, a1, b1, r0, r1, off0, off1, status, x0, y0, x1, y1, obs, F0,
                                  F1);
}

// The nodes beside the walls apart from the others.  A warp that holds a wall
// node runs the wall rule for its lane while the others wait, which in rows of
// a few warps costs as much again as the row (FP64: 390 operations against
// 134).  So the step kernels and the batched tiles give the border to blocks of
// its own and leave it out of the rows.
//
// By node pairs (PAIRS): the interior is (x0, x0 + 1) with x0 = 2, 4, ..., 2 npi
// (npi = floor((nx - 3) / 2): the pairs clear of the walls) and 1 <= y <= ny - 2,
// the border every other node: rows 0 and ny - 1, then the columns 0, 1 and 2
// npi + 2 .. nx - 1 of each inner row.  By nodes: the border is the wall nodes.
template <bool PAIRS> __host__ __device__ constexpr int border_columns(int nx) {
    return PAIRS ? nx - 2 * ((nx - 3) >> 1) : 2;
}
template <bool PAIRS> __host__ __device__ constexpr int border_count(int nx, int ny) {
    return 2 * nx + (ny - 2) * border_columns<PAIRS>(nx);
}
// Border node b in that order.
template <bool PAIRS> __device__ __forceinline__ void border_node(int b, int nx, int ny, int& x, int& y) {
    if (b < 2 * nx) {
        y = b < nx ? 0 : ny - 1;
        x = b < nx ? b : b - nx;
        return;
    }
    const int nbc = border_columns<PAIRS>(nx);
    const int k = b - 2 * nx;
    y = 1 + k / nbc;
    const int col = k - (y - 1) * nbc;
    x = col < (PAIRS ? 2 : 1) ? col : nx - nbc + col;
}

// Two fluid nodes from their pulled values (F0, F1: their frames in the frames'
// unit), FP32 and FP64 storage.  VEC: x-neighbours off1 = off0 + 1 with x0
// even, stored as pairs.
template <class T, bool FIELD, bool OBS, bool VEC>
__device__ __forceinline__ void core_fluid_pair(const Coef<typename T::R>& c, const Geom& gm, const Dst<T>& dst,
                                                const typename T::P* phi, typename T::R (&d0)[9],
                                                typename T::R (&h0)[5], typename T::R (&d1)[9],
                                                typename T::R (&h1)[5], typename T::R F0, typename T::R F1, int x0,
                                                int y0, int x1, int y1, int* status, double* obs) {
    using R = typename T::R;
    constexpr bool FR = Framed<T>::value;
    const Coll<R>& k = c.k;
    const int off0 = y0 * gm.pitch + x0, off1 = y1 * gm.pitch + x1;
    R phi0 = R(1), phi1 = R(1);
    if constexpr (FIELD) {
        if (in_plane(gm, off0)) phi0 = Conv<typename T::P, R>::ld(VEC ? at(phi, 0, off0) : phi + off0);
        if (in_plane(gm, off1)) phi1 = Conv<typename T::P, R>::ld(VEC ? at(phi, 1, off0) : phi + off1);
    }
    typename FrameStore<T>::type k0, k1;
    R l0, l1, t0, t1;  // T - T0 - F and T - T0 of both nodes
    if constexpr (std::is_same<R, float>::value) {
        // both nodes in paired instructions
        F2 d[9], h[5], next;
#pragma unroll
        for (int i = 0; i < 9; ++i) d[i] = F2(d0[i], d1[i]);
#pragma unroll
        for (int j = 0; j < 5; ++j) h[j] = F2(h0[j], h1[j]);
        const F2 F(F0, F1);
        const Por<F2> p = por_of<F2, FIELD>(k, F2(phi0, phi1));
        const Sums<F2> s = sums_of(d, h);
        const Vel<F2> v = velocity<F2, FR, FIELD>(k, p, s, op::mul(k.fu, F));
        if (too_fast(v)) atomicOr(status, 1);
        F2 shift(0.f, 0.f);
        if constexpr (FR) shift = frame_next<T>(k, v.dT, F, next, k0, k1);
        collide_fluid<F2, FIELD, FR>(k, p, s, v, shift, d, h);
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            d0[i] = d[i].v.x;
            d1[i] = d[i].v.y;
        }
#pragma unroll
        for (int j = 0; j < 5; ++j) {
            h0[j] = h[j].v.x;
            h1[j] = h[j].v.y;
        }
        l0 = v.dTl.v.x;
        l1 = v.dTl.v.y;
        t0 = v.dT.v.x;
        t1 = v.dT.v.y;
    } else {
        // one after the other
        auto node = [&](R (&d)[9], R (&h)[5], R F, R phi_n, typename FrameStore<T>::type& code, R& l, R& t) {
            const Por<R> p = por_of<R, FIELD>(k, phi_n);
            const Sums<R> s = sums_of(d, h);
            const Vel<R> v = velocity<R, FR, FIELD>(k, p, s, op::mul(F, k.fu));
            if (too_fast(v)) atomicOr(status, 1);
            R next;
            collide_fluid<R, FIELD, FR>(k, p, s, v, frame_next<T>(k, v.dT, F, next, code), d, h);
            l = v.dTl;
            t = v.dT;
        };
        node(d0, h0, F0, phi0, k0, l0, t0);
        node(d1, h1, F1, phi1, k1, l1, t1);
    }
    if constexpr (VEC) {
        if (in_plane(gm, off0, 2)) {
            if constexpr (FR) frame_st2<T>(at(dst.t, 0, off0), k0, k1);
#pragma unroll
            for (int i = 0; i < 9; ++i) Conv2<typename T::SF, R, T::cg>::st(at(dst.f, i * gm.plane, off0), d0[i], d1[i]);
#pragma unroll
            for (int j = 0; j < 5; ++j) Conv2<typename T::SG, R, T::cg>::st(at(dst.g, j * gm.plane, off0), h0[j], h1[j]);
        }
    } else if (in_plane(gm, off0) && in_plane(gm, off1)) {
        if constexpr (FR) {
            dst.t[off0] = k0;
            dst.t[off1] = k1;
        }
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            Conv<typename T::SF, R, T::cg>::st(dst.f + i * gm.plane + off0, d0[i]);
            Conv<typename T::SF, R, T::cg>::st(dst.f + i * gm.plane + off1, d1[i]);
        }
#pragma unroll
        for (int j = 0; j < 5; ++j) {
            Conv<typename T::SG, R, T::cg>::st(dst.g + j * gm.plane + off0, h0[j]);
            Conv<typename T::SG, R, T::cg>::st(dst.g + j * gm.plane + off1, h1[j]);
        }
    }
    if constexpr (OBS) {
        obs_put(gm, obs, x0, y0, FR ? (double)op::mul(F0, k.fu) + (double)l0 : (double)t0);
        obs_put(gm, obs, x1, y1, FR ? (double)op::mul(F1, k.fu) + (double)l1 : (double)t1);
    }
}

// Two nodes at once: when both are fluid nodes all 28 loads are issued before
// any arithmetic (twice the bytes in flight of one node per thread); nodes
// outside the lattice (valid = false) or on walls take the one-node path.
template <class T, bool FIELD, bool OBS = false>
__device__ __forceinline__ void update_pair(const CoefOf<T>& c, const Geom& gm, const Src<T>& src,
                                            const Dst<T>& dst, const typename T::P* phi, int x0, int y0,
                                            bool v0, int x1, int y1, bool v1, int* status, double* obs = nullptr) {
    using R = typename T::R;
    const bool f0 = v0 && x0 > 0 && x0 < gm.nx - 1 && y0 > 0 && y0 < gm.ny - 1;
    const bool f1 = v1 && x1 > 0 && x1 < gm.nx - 1 && y1 > 0 && y1 < gm.ny - 1;
    if (f0 && f1) {
        if constexpr (Core<T>::value) {
            R d0[9], h0[5], d1[9], h1[5];
            const int off0 = y0 * gm.pitch + x0, off1 = y1 * gm.pitch + x1;
            pull<T>(src, gm, off0, d0, h0);
            pull<T>(src, gm, off1, d1, h1);
            const R F0 = core_frame_in<T>(c.k, src, gm, off0, h0);
            const R F1 = core_frame_in<T>(c.k, src, gm, off1, h1);
            core_fluid_pair<T, FIELD, OBS, false>(c, gm, dst, phi, d0, h0, d1, h1, F0, F1, x0, y0, x1, y1, status,
                                                  obs);
        } else {
            update_fluid_pair_x2<T, FIELD, OBS>(c, gm, src, dst, phi, x0, y0, x1, y1, status, obs);
        }
        return;
    }
    if (v0) update_node<T, FIELD, OBS>(c, gm, src, dst, phi, x0, y0, status, obs);
    if (v1) update_node<T, FIELD, OBS>(c, gm, src, dst, phi, x1, y1, status, obs);
}

// The fluid nodes (x0, y) and (x0 + 1, y), x0 even (FP32 and FP64 storage).
template <class T, bool FIELD, bool OBS = false>
__device__ __forceinline__ void update_fluid_xpair(const Coef<typename T::R>& c, const Geom& gm, const Src<T>& src,
                                                   const Dst<T>& dst, const typename T::P* phi, int x0, int y,
                                                   int* status, double* obs = nullptr) {
    using R = typename T::R;
    R d0[9], h0[5], d1[9], h1[5], F0, F1;
    pull_x2<T>(src, gm, y * gm.pitch + x0, d0, h0, d1, h1);
    core_frame_in_x2<T>(c.k, src, gm, y * gm.pitch + x0, h0, h1, F0, F1);
    core_fluid_pair<T, FIELD, OBS, true>(c, gm, dst, phi, d0, h0, d1, h1, F0, F1, x0, y, x0 + 1, y, status, obs);
}

// Two nodes side by side, (x0, y) and (x0 + 1, y) with x0 even: when both are
// fluid nodes the populations with e_x = 0, the stores and the frames move
// as aligned pairs (about a third fewer memory instructions than two nodes
// apart); otherwise each valid node takes the one-node path.
template <class T, bool FIELD, bool OBS = false>
__device__ __forceinline__ void update_xpair(const CoefOf<T>& c, const Geom& gm, const Src<T>& src,
                                             const Dst<T>& dst, const typename T::P* phi, int x0, int y,
                                             int* status, double* obs = nullptr) {
    using R = typename T::R;
    const int x1 = x0 + 1;
    if (x0 > 0 && x1 < gm.nx - 1 && y > 0 && y < gm.ny - 1) {
        if constexpr (Core<T>::value) {
            update_fluid_xpair<T, FIELD, OBS>(c, gm, src, dst, phi, x0, y, status, obs);
        } else {
            const int off0 = y * gm.pitch + x0, off1 = off0 + 1;
            R d0[9], h0[5], d1[9], h1[5];
            pull_x2<T>(src, gm, off0, d0, h0, d1, h1);
            R F0 = R(0), F1 = R(0);
            frame_in_x2<T>(c, src, gm, off0, h0, h1, F0, F1);
            const Drag<R> dr0 = drag_at<R, FIELD, typename T::P>(c, gm, phi, off0);
            const Drag<R> dr1 = drag_at<R, FIELD, typename T::P>(c, gm, phi, off1);
            collide_fluid_pair_x2<T, OBS, true>(c, gm, dst, d0, h0, d1, h1, dr0, dr1, off0, off1, status, x0, y, x1,
                                                y, obs, F0, F1);
        }
        return;
    }
    if (x0 < gm.nx) update_node<T, FIELD, OBS>(c, gm, src, dst, phi, x0, y, status, obs);
    if (x1 < gm.nx) update_node<T, FIELD, OBS>(c, gm, src, dst, phi, x1, y, status, obs);
}

// T - T0 of the post-stream state at node (x, y), pulled from B_{n-1}
// (the wall rule's temperature on wall nodes), in FP64 (framed storage adds
// the frame to the local part in FP64, so the value keeps its precision).
template <class T>
__device__ __forceinline__ double node_dT(const CoefOf<T>& c, const Geom& gm, const Src<T>& prev, int x,
                                          int y) {
    using R = typename T::R;
    const Normal nr = normal_of(gm, x, y);
    if constexpr (Framed<T>::value) {
        R F;
        if (nr.dx == 0 && nr.dy == 0) {
            const R l = pull_heat<T>(c, prev, gm, y * gm.pitch + x, F) + c.qhalf;
            return (double)F + (double)l;
        }
        if (gm.thermal_bc == 1) return (double)c.dTc;
        if (nr.dx != 0) return (double)(x == 0 ? c.dTh : c.dTc);
        const R lf = pull_heat<T>(c, prev, gm, (y + nr.dy) * gm.pitch + x, F) + c.qhalf;
        if (gm.adi_order == 2) {
            R Fff;
            const R lff = pull_heat<T>(c, prev, gm, (y + 2 * nr.dy) * gm.pitch + x, Fff) + c.qhalf;
            return (4.0 * ((double)F + (double)lf) - ((double)Fff + (double)lff)) / 3.0;
        }
        return (double)F + (double)lf;
    } else {
        R F;
        if (nr.dx == 0 && nr.dy == 0) return (double)(pull_heat<T>(c, prev, gm, y * gm.pitch + x, F) + c.qhalf);
        if (gm.thermal_bc == 1) return (double)c.dTc;
        if (nr.dx != 0) return (double)(x == 0 ? c.dTh : c.dTc);
        const R dTf = pull_heat<T>(c, prev, gm, (y + nr.dy) * gm.pitch + x, F) + c.qhalf;
        if (gm.adi_order == 2) {
            const R dTff = pull_heat<T>(c, prev, gm, (y + 2 * nr.dy) * gm.pitch + x, F) + c.qhalf;
            return (double)((R(4) * dTf - dTff) * R(1.0 / 3.0));
        }
        return (double)dTf;
    }
}

// node_dT of node (x, y), x = k (k < 5) or nx - 1 - (k - 5), from the wall
// columns an observing step stored (obs_put): the stored value off the walls;
// on the walls the wall rule's temperature, imposed on the vertical walls and,
// on the adiabatic rows, taken from the stored rows next to them in the
// arithmetic node_dT uses, so both give the same bits.
template <class T>
__device__ __forceinline__ double obs_dT(const CoefOf<T>& c, const Geom& gm, const double* obs, int k,
                                         int y) {
    using R = typename T::R;
    const int x = k < 5 ? k : gm.nx - 1 - (k - 5);
    const Normal nr = normal_of(gm, x, y);
    if (nr.dx == 0 && nr.dy == 0) return obs[kObsCols * y + k];
    if (gm.thermal_bc == 1) return (double)c.dTc;
    if (nr.dx != 0) return (double)(x == 0 ? c.dTh : c.dTc);
    const double tf = obs[kObsCols * (y + nr.dy) + k];
    if (gm.adi_order == 2) {
        const double tff = obs[kObsCols * (y + 2 * nr.dy) + k];
        if constexpr (Framed<T>::value)
            return (4.0 * tf - tff) / 3.0;
        else
            return (double)((R(4) * R(tf) - R(tff)) * R(1.0 / 3.0));
    }
    return tf;
}

// Non-negative values as integers: the order of the bit patterns is that of the
// values, with NaN (of either sign) above infinity, so that a maximum over a
// lattice that holds a NaN is NaN; and integers stay off the FP64 unit.
__device__ __forceinline__ unsigned order_bits(float v) { return __float_as_uint(v); }
__device__ __forceinline__ unsigned long long order_bits(double v) { return (unsigned long long)__double_as_longlong(v); }
__device__ __forceinline__ double from_order(unsigned b) { return (double)__uint_as_float(b); }
__device__ __forceinline__ double from_order(unsigned long long b) { return __longlong_as_double((long long)b); }

// Block-wide max, max (non-negative), sum, sum of four doubles per thread; the
// result in thread 0.  256 threads.  The threads' values meet in shared memory
// and one warp folds them, eight per lane and then across the lanes: 26
// FP64 instructions per block for the sums, where a butterfly in every warp
// takes 90 (an FP64 warp instruction takes an SM 16 cycles).
__device__ __forceinline__ void fold_block(double (&v)[4], double (*sh)[256]) {
    const int t = threadIdx.x;
#pragma unroll
    for (int k = 0; k < 4; ++k) sh[k][t] = v[k];
    __syncthreads();
    if (t < 32) {
        unsigned long long m0 = order_bits(v[0]), m1 = order_bits(v[1]);
#pragma unroll
        for (int w = 1; w < 8; ++w) {
            m0 = max(m0, order_bits(sh[0][t + 32 * w]));
            m1 = max(m1, order_bits(sh[1][t + 32 * w]));
            v[2] += sh[2][t + 32 * w];
            v[3] += sh[3][t + 32 * w];
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            m0 = max(m0, __shfl_xor_sync(0xffffffffu, m0, o));
            m1 = max(m1, __shfl_xor_sync(0xffffffffu, m1, o));
            v[2] += __shfl_xor_sync(0xffffffffu, v[2], o);
            v[3] += __shfl_xor_sync(0xffffffffu, v[3], o);
        }
        v[0] = from_order(m0);
        v[1] = from_order(m1);
    }
}

// 12 dT/dx (Eq. 38's one-sided five-point derivative, times the spacing) at both
// ends of a row from the five temperatures next to each wall.
__device__ __forceinline__ double slope_hot(const double (&t)[5]) {
    return -25.0 * t[0] + 48.0 * t[1] - 36.0 * t[2] + 16.0 * t[3] - 3.0 * t[4];
}
__device__ __forceinline__ double slope_cold(const double (&t)[5]) {
    return 25.0 * t[0] - 48.0 * t[1] + 36.0 * t[2] - 16.0 * t[3] + 3.0 * t[4];
}

// Mean Nusselt numbers (Eq. 38) of both vertical walls over a whole block of 256
// threads (valid in thread 0): Nu(y) = -L dT/dx / dT, trapezoidal mean over y,
// FP64.
template <class T>
__device__ __forceinline__ void nusselt_block(const CoefOf<T>& c, const Geom& gm, const Src<T>& prev,
                                              double L, double dT, double (*sh)[256], double* nu_hot,
                                              double* nu_cold) {
    double w[4] = {0.0, 0.0, 0.0, 0.0};
    for (int y = threadIdx.x; y < gm.ny; y += 256) {
        double tl[5], tr[5];
#pragma unroll
        for (int k = 0; k < 5; ++k) {
            tl[k] = (double)node_dT<T>(c, gm, prev, k, y);
            tr[k] = (double)node_dT<T>(c, gm, prev, gm.nx - 1 - k, y);
        }
        const double wt = (y == 0 || y == gm.ny - 1) ? 0.5 : 1.0;
        w[2] += wt * slope_hot(tl);
        w[3] += wt * slope_cold(tr);
    }
    fold_block(w, sh);
    const double scale = -L / (12.0 * dT) / (double)(gm.ny - 1);
    *nu_hot = w[2] * scale;
    *nu_cold = w[3] * scale;
}

}  // namespace lbm
