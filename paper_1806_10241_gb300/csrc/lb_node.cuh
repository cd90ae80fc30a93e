// The node update (sources, collisions, back-transform) on a type V with +, -,
// *, fma2(a, b, c) = a b + c, rcp2(a) = 1 / a, V::of(constant), V::lit(number)
// and V::unit(constant, number), whichever of the two is cheaper for the type:
// pairs of FP32 nodes (F2) or one FP64 node (D1).  Included inside the namespace
// that holds those types.
//
// No sum or difference here has a product as an operand, but for products with
// a power of two, which are exact: where a product is added, fma2 says so.
// Otherwise the assembler would decide product by product, and differently
// where the update is inlined into another kernel, whether the product is
// rounded before it is added (it fuses packed operations in spite of
// -fmad=false), and paths that promise the same bits would rest on that.
#ifndef LB_NODE_FN
#define LB_NODE_FN __device__ __forceinline__
#endif

// Plane indices
enum { F0 = 0, G0 = 9, H0 = 14 };

// Parameters of the node update as its operands: in FP32 as packed pairs with
// equal halves, which the packed instructions take as they lie in the
// parameters, where a scalar would first be copied into a pair.
template <typename E> struct NodeConst {
    E rho0, T0, bfx, fb, nu, nuh, alh, k3;              // fb = rho0 g_beta; nu / 2, alpha / 2, rho0 / 3
    // relaxation and back-transform factors (n..: the negative), storage scale, 1, -1
    E c3, c4, nc4, ch, nch, cg, ct, m9, m6, m5, sg, os, one, mone;
};

template <class V> struct NodeVals {
    V v[NQ];  // f, g, h
};

// The factors of a column's geometric sources, from iy = 1 / y, or 0 in the
// planar form (no geometric sources).
template <class V> struct Geo {
    V gy, ngy, nuiyh, nuiy, alhiy, niy2nu, m2iy2nu;
};
template <class V, class NC> LB_NODE_FN Geo<V> geo_of(const NC &c, V iy)
{
    Geo<V> g;
    g.gy = iy;
    g.ngy = iy * V::unit(c.mone, -1.0);
    g.nuiyh = iy * V::of(c.nuh);
    g.nuiy = iy * V::of(c.nu);
    g.alhiy = iy * V::of(c.alh);
    g.niy2nu = g.nuiy * g.ngy;
    g.m2iy2nu = g.niy2nu * V::lit(2.0);
    return g;
}

// The gradient inputs are the undivided central differences (twice the
// derivatives); the halves are folded into the geometric factors, which is
// exact.
// kScale: the post-collision values come out multiplied by osc, a power of two
// (the FP16 storage scale): osc is folded into the constants of the
// post-collision moments and into the fused multiply-add that adds them to
// the streamed values.  Scaling by a power of two commutes with every
// rounding, so the results are exactly osc times the unscaled ones.
//
// What the order of the terms is chosen for: packed instructions occupy the
// FP32 pipe for two cycles and are two thirds of its work, so factors of +-1
// and +-2 ride on the velocities (n2ux, nuy, ...) instead of costing a
// multiplication per product, and products with rho are taken from the
// momentum (rho ux^2 = jx ux): 267 packed operations per pair and three
// reciprocals.  On one-step launches of 1024 x 2048 this and the bare reciprocal
// (rcp1) took 53.4 -> 52.0 us in FP32 and 49.2 -> 45.7 us in FP16 against the
// terms as update_pinned has them.
template <bool kScale, class V, class NC>
LB_NODE_FN void update_node2(const NC &c, bool explicit_src, const Geo<V> &geo, const V fv[9], const V gv[5],
                             const V hv[5], V dxuy, V dyux, V dyuy, V dyut, V dyT, NodeVals<V> &o)
{
    const V OS = V::of(c.os), one = V::unit(c.one, 1.0), mone = V::unit(c.mone, -1.0);
    auto plus = [&](V v, V m) { return kScale ? fma2(v, OS, m) : v + m; };
    // sum and difference with a product p.  The units are constants of the
    // parameters in FP32 (as literals they take two more registers, and the FP32
    // strips spill: 1024 x 2048 42.5 us per step, 40.6 so), literals in FP64
    // (where they cost nothing: 256 x 512 87.8 us per step, 89.1 as constants).
    // All this costs small FP32 tiles 1 % (100 x 100: 2.37 -> 2.40 us per step).
    auto add_p = [&](V a, V p) { return fma2(p, one, a); };
    auto sub_p = [&](V a, V p) { return fma2(p, mone, a); };
    auto plus_p = [&](V v, V p) { return fma2(v, OS, p); };

    // output moments, Eq. 18, 35, 47 (deviation form)
    const V a57 = fv[5] - fv[7], a86 = fv[8] - fv[6];
    const V s57 = fv[5] + fv[7], s68 = fv[6] + fv[8];
    const V s13 = fv[1] + fv[3], s24 = fv[2] + fv[4];
    const V s5678 = s57 + s68;
    const V rdo = (fv[0] + s13) + (s24 + s5678);
    const V Dxxy = a57 - a86, Dxyy = a57 + a86;
    const V jxo = (fv[1] - fv[3]) + Dxyy;
    const V jyo = (fv[2] - fv[4]) + Dxxy;
    const V pso = (gv[0] + gv[1]) + (gv[2] + gv[3]) + gv[4];
    const V tdo = (hv[0] + hv[1]) + (hv[2] + hv[3]) + hv[4];

    // sources at the pre-collision state, two sweeps (see update_node)
    const V gy = geo.gy, ngy = geo.ngy, niy2nu = geo.niy2nu, m2iy2nu = geo.m2iy2nu;
    const V Gx = (dxuy + dyux) * geo.nuiyh;
    const V Gy = dyuy * geo.nuiy;
    const V Gw = dyut * geo.nuiyh;
    const V Gt = dyT * geo.alhiy;
    const V Fbx = V::of(c.bfx);
    const V Fb = V::of(c.fb), rho0 = V::of(c.rho0), T0 = V::of(c.T0), half = V::lit(0.5);
    V rd = rdo, jx = jxo, jy = jyo, ps = pso, td = tdo;
    V MA, Fx, Fy, Sps, Sph;
    auto sweep = [&]() {
        const V r = rho0 + rd, ir = rcp2(r);
        const V uyyn = (jy * ir) * ngy;  // -u_y / y
        Fx = fma2(Fb, td, fma2(jx, uyyn, fma2(r, Gx, Fbx)));
        Fy = fma2(jy, m2iy2nu, fma2(r, Gy, ((ps - jy) * (ps + jy)) * (ir * gy)));
        Sps = fma2(ps, fma2(uyyn, V::lit(2.0), niy2nu), r * Gw);
        Sph = fma2(uyyn, T0 + td, Gt);
        jx = fma2(Fx, half, jxo);
        jy = fma2(Fy, half, jyo);
        ps = fma2(Sps, half, pso);
        td = fma2(Sph, half, tdo);
        MA = jy * ngy;
        rd = fma2(MA, half, rdo);
    };
    sweep();
    if (explicit_src) {
        MA = jyo * ngy;
        rd = fma2(MA, half, rdo);
    } else {
        sweep();
    }
    const V r = rho0 + rd, ir = rcp2(r);
    const V ux = jx * ir, uy = jy * ir;
    const V phi = T0 + td;

    // D2Q9 cascaded collision, Eq. 17
    const V Dxx = s13 + s5678, Dyy = s24 + s5678;
    const V Dxy = s57 - s68, Dxxyy = s5678;
    const V k3 = V::of(c.k3);
    const V Kxx = k3 + Dxx, Kyy = k3 + Dyy;
    const V ux2 = ux * ux, uy2 = uy * uy;
    const V rxx = jx * ux, ryy = jy * uy;  // rho ux^2, rho uy^2
    const V nux = ux * mone, nuy = uy * mone, n2ux = ux * V::lit(-2.0), n2uy = uy * V::lit(-2.0);
    const V uxy4 = n2ux * n2uy;
    const V p3 = (fma2(rd, V::lit(2.0 / 3.0), fma2(jx, ux, ryy)) - (Dxx + Dyy)) * V::of(c.c3);
    const V c4 = V::of(c.c4), ch = V::of(c.ch), nch = V::of(c.nch);
    const V p4 = (fma2(jy, nuy, rxx) - (Dxx - Dyy)) * c4;
    const V nx5 = fma2(jx, nuy, Dxy);  // -(rho ux uy - Dxy)
    const V p5 = nx5 * V::of(c.nc4), np5 = nx5 * c4;
    // -(3 p3 + p4) / 2 and -(3 p3 - p4) / 2
    const V hp = fma2(p3, V::lit(-1.5), p4 * V::lit(-0.5)), hm = fma2(p3, V::lit(-1.5), p4 * half);
    const V rxx2 = rxx * V::lit(2.0), ryy2 = ryy * V::lit(2.0);
    // p6: (2 r ux^2 uy + Dxxy - 2 ux Dxy - uy Kxx) omhi/4 - uy (3 p3 + p4)/2 - 2 ux p5
    const V Z = fma2(nuy, Kxx, fma2(n2ux, Dxy, fma2(rxx2, uy, Dxxy)));
    const V p6 = fma2(Z, ch, fma2(uy, hp, n2ux * p5));
    const V Y = fma2(nux, Kyy, fma2(n2uy, Dxy, fma2(ryy2, ux, Dxyy)));
    const V p7 = fma2(Y, ch, fma2(ux, hm, n2uy * p5));
    // p8
    V B = fma2(ux2, Kyy, Dxxyy);
    B = fma2(uy2, Kxx, B);
    B = fma2(uxy4, Dxy, B);
    B = fma2(n2ux, Dxyy, B);
    B = fma2(n2uy, Dxxy, B);
    const V Wm = fma2(rd, V::lit(1.0 / 9.0), (rxx2 * uy2) * V::lit(1.5)) - B;
    V p8 = fma2(p3, V::lit(-2.0), Wm * ch);
    p8 = fma2(uy2, hp, p8);
    p8 = fma2(ux2, hm, p8);
    p8 = fma2(uxy4, np5, p8);
    p8 = fma2(n2uy, p6, p8);
    p8 = fma2(n2ux, p7, p8);
    // source moments, Eq. 26
    const V p0 = MA * V::of(c.m9), p1 = Fx * V::of(c.m6), p2 = Fy * V::of(c.m6);
    // back-transform, Eq. 27, grouped
    {
        const V A0 = sub_p(p0, p3);
        const V E = fma2(p8, V::lit(-2.0), add_p(A0, p4)), Fm = fma2(p8, V::lit(-2.0), sub_p(A0, p4));
        const V u = fma2(p7, V::lit(2.0), p1), w = fma2(p6, V::lit(2.0), p2);
        o.v[0] = fma2(sub_p(p8, p3), V::lit(4.0), plus_p(fv[0], p0));
        o.v[1] = plus(fv[1], E) + u;
        o.v[3] = plus(fv[3], E) - u;
        o.v[2] = plus(fv[2], Fm) + w;
        o.v[4] = plus(fv[4], Fm) - w;
        const V B0 = fma2(p3, V::lit(2.0), add_p(p8, p0));
        const V C5 = sub_p(B0, np5), C6 = sub_p(B0, p5);
        const V n17 = sub_p(p7, p1), n26 = sub_p(p6, p2);
        const V us = n17 + n26, vd = n17 - n26;
        o.v[5] = plus(fv[5], C5) - us;
        o.v[7] = plus(fv[7], C5) + us;
        o.v[6] = plus(fv[6], C6) + vd;
        o.v[8] = plus(fv[8], C6) - vd;
    }

    // D2Q5 cascaded collisions, Eq. 34 / 49 (sign reading of the paper: -),
    // the bracket of q3, q4 with its sign turned
    const V uu = fma2(ux, ux, uy2), ud = fma2(nuy, uy, ux2);
    const V sg = V::of(c.sg);
    const V ncu = fma2(sg, uu, V::lit(-2.0 / 3.0)), ncd = sg * ud;
    const V m5 = V::of(c.m5);
    {
        const V kxn = gv[3] - gv[1], kyn = gv[4] - gv[2];  // -kappa'_x, -kappa'_y
        const V kxx = gv[1] + gv[3], kyy = gv[2] + gv[4];
        const V cg = V::of(c.cg);
        const V q1 = fma2(ps, ux, kxn) * cg;
        const V q2 = fma2(ps, uy, kyn) * cg;
        const V X3 = fma2(ps, ncu, fma2(fma2(ux, kxn, uy * kyn), V::lit(2.0), kxx + kyy));
        const V X4 = fma2(ps, ncd, fma2(fma2(ux, kxn, nuy * kyn), V::lit(2.0), kxx - kyy));
        const V q3 = fma2(X3, nch, fma2(ux, q1, uy * q2));
        const V q4 = fma2(X4, nch, fma2(ux, q1, nuy * q2));
        const V q0 = Sps * m5, Q = add_p(q3, q0), Qp = Q + q4, Qm = Q - q4;
        o.v[G0 + 0] = fma2(q3, V::lit(-4.0), plus_p(gv[0], q0));
        o.v[G0 + 1] = add_p(plus(gv[1], Qp), q1);
        o.v[G0 + 3] = sub_p(plus(gv[3], Qp), q1);
        o.v[G0 + 2] = add_p(plus(gv[2], Qm), q2);
        o.v[G0 + 4] = sub_p(plus(gv[4], Qm), q2);
    }
    {
        const V kxn = hv[3] - hv[1], kyn = hv[4] - hv[2];
        const V Hxx = hv[1] + hv[3], Hyy = hv[2] + hv[4];
        const V ct = V::of(c.ct);
        const V r1 = fma2(phi, ux, kxn) * ct;
        const V r2 = fma2(phi, uy, kyn) * ct;
        // 2 c^2 phi - (kxx + kyy) with the rest parts written out: 2/3 td - (Hxx + Hyy)
        const V X3 = fma2(V::lit(-2.0 / 3.0), td, fma2(phi, sg * uu, fma2(fma2(ux, kxn, uy * kyn), V::lit(2.0), Hxx + Hyy)));
        const V X4 = fma2(phi, ncd, fma2(fma2(ux, kxn, nuy * kyn), V::lit(2.0), Hxx - Hyy));
        const V r3 = fma2(X3, nch, fma2(ux, r1, uy * r2));
        const V r4 = fma2(X4, nch, fma2(ux, r1, nuy * r2));
        const V r0 = Sph * m5, Q = add_p(r3, r0), Qp = Q + r4, Qm = Q - r4;
        o.v[H0 + 0] = fma2(r3, V::lit(-4.0), plus_p(hv[0], r0));
        o.v[H0 + 1] = add_p(plus(hv[1], Qp), r1);
        o.v[H0 + 3] = sub_p(plus(hv[3], Qp), r1);
        o.v[H0 + 2] = add_p(plus(hv[2], Qm), r2);
        o.v[H0 + 4] = sub_p(plus(hv[4], Qm), r2);
    }
}
