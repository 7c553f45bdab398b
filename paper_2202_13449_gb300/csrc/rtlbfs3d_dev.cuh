// rtlbfs3d_dev.cuh -- the per-face arithmetic of 3D RTLBFS (arXiv
// 2202.13449, Section 3.2 with the D3Q19 lattice of Eqs. 5-6), templated on
// the value type V (float, double, or a host counting type).
//
// A face is handled in its own frame: normal n (index 0) and two tangents
// t1, t2 (indices 1, 2).  Cell quantities enter as (drho, u_n, u_t1, u_t2,
// tau) with drho = rho - 1 and tau = T - Tbar, Tbar a face reference
// temperature, so FP32 never differences the O(1) parts of rho and rho T;
// the constant c_s^2 of the normal momentum flux is dropped (it cancels in
// the flux divergence of a closed cell).
#pragma once

#include "rtlbfs_dev.cuh"

namespace rtlbfs3 {

using rtlbfs::FaceLine;
using rtlbfs::vfma;
using rtlbfs::vtraits;

// One cell seen from a face: values and gradients along n, t1, t2.
template <typename V>
struct CellNT3 {
    V q[5];
    V gn[5];
    V g1[5];
    V g2[5];
};

// Eq. 29, Eqs. 46-48 and the braces of Eqs. 57-59 for one face.
//
// Nodes.  Node (a, b, c) of the D3Q19 lattice sits at x_S + (a n + b t1 +
// c t2) h.  A cell's reconstruction plane restricted to a column a = const
// is linear in (b, c), so each primitive on column a is C + b S1 + c S2:
// a = -1 the left plane, a = +1 the right plane, a = 0 their mean (Eq. 29).
// The 19 nodes are the centre, the axis nodes +-e_a and the edge nodes
// +-e_a +-e_b (a < b).  With products formed at the nodes, the lattice
// differences
//   d_a f  = f(+e_a) - f(-e_a)                   = 2 h D_a f
//   dd_a f = f(+e_a) - 2 f(0) + f(-e_a)          = h^2 D_aa f
//   dd_ab f = f(+a+b) - f(+a-b) - f(-a+b) + f(-a-b) = 4 h^2 D_ab f
// turn Eqs. 46-48 into (the powers of h cancel)
//   drho* = drho - 1/2 sum_a d_a m_a + 1/2 sum_a dd_a (m_a u_a + cs2 drho)
//           + 1/4 sum_{a<b} dd_ab (m_a u_b)
//   m_a*  = m_a - 1/2 sum_b d_b X_ab
//           + cs2/2 [sum_b dd_b m_a + 2 dd_a m_a + 1/2 sum_{b!=a} dd_ab m_b]
//   e*    = e - 1/2 sum_a (Tbar d_a m_a + d_a (m_a tau)) + cs2/2 sum_a dd_a e
// with m_a = rho u_a, X_ab = m_a u_b + cs2 drho delta_ab, e = rho T - Tbar.
// keep = 1 on an interior face, 0 on a wall face whose tangential velocity
// is (uw1, uw2), 0 on an interior face: no mass through the wall,
// (rho u_t)* = rho* u_wall,t.
// F = (mass, n-, t1-, t2-momentum, energy) flux along +n.
//
// The products are never formed node by node.  On a column they are
// polynomials in (b, c) of degree <= 3, and a lattice difference picks
// coefficients of one of them:
//   d_t f   = 2 (odd part in t at a = 0),  dd_t f = 2 (t^2 coefficient),
//   dd_t1t2 f = 4 (b c coefficient),
//   dd_nt f = 2 (odd part in t on a = +1, minus that on a = -1):
// the same numbers with a third fewer operations (281 a face against 435
// for products at the 19 nodes), and without the cancellation of the node
// differences.  FP64 runs at the FMA rate, so there the step follows the
// count: 20 steps of an 80^3 mesh and the download, FP64, 34.8 -> 29.5 ms with
// the step kernel of that time.
//
// The first stage, face3_columns, forms the coefficients C, S1, S2 of the
// five primitives on the three columns (A: a = -1, M: a = 0, B: a = +1);
// face_flux3_columns does the rest.
template <typename V>
struct Cols3 {
    V A[5], A1[4], A2[4];
    V M[5], M1[5], M2[5];
    V B[5], B1[4], B2[4];
};

template <typename V>
__host__ __device__ __forceinline__ void face3_columns(const CellNT3<V>& L, const CellNT3<V>& Rc,
                                                      const FaceLine<V>& fl, Cols3<V>& c)
{
    using T = vtraits<V>;
    const V half = T::bc(0.5);
    const V h = fl.h;
    const V wL = fl.cL + h, mwR = fl.cR - h;  // wL, -wR: centre-to-face distances
    const V hh = h * half;
#pragma unroll
    for (int k = 0; k < 5; ++k) {
        c.A[k] = vfma(L.gn[k], fl.cL, L.q[k]);
        c.B[k] = vfma(Rc.gn[k], fl.cR, Rc.q[k]);
        if (k < 4) {  // the side columns' temperature slopes enter nowhere
            c.A1[k] = L.g1[k] * h;
            c.A2[k] = L.g2[k] * h;
            c.B1[k] = Rc.g1[k] * h;
            c.B2[k] = Rc.g2[k] * h;
        }
        c.M[k] = half * (vfma(L.gn[k], wL, L.q[k]) + vfma(Rc.gn[k], mwR, Rc.q[k]));
        c.M1[k] = hh * (L.g1[k] + Rc.g1[k]);
        c.M2[k] = hh * (L.g2[k] + Rc.g2[k]);
    }
}

// What a side column (a = -1 or +1) contributes: centre values and the odd
// parts in t1 and t2 that the cross differences need.
template <typename V>
struct SideCol3 {
    V m[3];        // rho u_n, rho u_1, rho u_2
    V e;           // rho T - Tbar
    V ln1, l11;    // linear in t1: rho u_n, rho u_1
    V ln2, l22;    // linear in t2: rho u_n, rho u_2
    V o1, o2;      // odd parts: rho u_n u_1 in t1, rho u_n u_2 in t2
};

template <typename V>
__host__ __device__ __forceinline__ SideCol3<V> side_column3(const V C[5], const V S1[4],
                                                            const V S2[4], V Tbar)
{
    SideCol3<V> s;
    const V r = vtraits<V>::bc(1.0) + C[0];
#pragma unroll
    for (int a = 0; a < 3; ++a) s.m[a] = vfma(C[0], C[1 + a], C[1 + a]);
    s.e = vfma(C[0], Tbar + C[4], C[4]);
    s.ln1 = vfma(r, S1[1], S1[0] * C[1]);
    s.l11 = vfma(r, S1[2], S1[0] * C[2]);
    s.o1 = vfma(S1[2], vfma(S1[0], S1[1], s.m[0]), s.ln1 * C[2]);
    s.ln2 = vfma(r, S2[1], S2[0] * C[1]);
    s.l22 = vfma(r, S2[3], S2[0] * C[3]);
    s.o2 = vfma(S2[3], vfma(S2[0], S2[1], s.m[0]), s.ln2 * C[3]);
    return s;
}

// wall(mn, m1, m2, rho): the wall rule on the predicted momenta.
template <typename V, class W>
__host__ __device__ __forceinline__ void face_flux3_wall(const Cols3<V>& c, V Tbar,
                                                        const FaceLine<V>& fl, W wall, V F[5])
{
    using T = vtraits<V>;
    const V zero = T::bc(0.0), half = T::bc(0.5), one = T::bc(1.0);
    const V two = T::bc(2.0), three = T::bc(3.0), six = T::bc(6.0);
    const V m2 = T::bc(-2.0), mhalf = T::bc(-0.5);
    const V cs2 = T::bc(1.0 / 3.0), mcs2 = T::bc(-1.0 / 3.0), hcs2 = T::bc(0.5 / 3.0);

    const SideCol3<V> a = side_column3(c.A, c.A1, c.A2, Tbar);
    const SideCol3<V> b = side_column3(c.B, c.B1, c.B2, Tbar);
    // differences along the normal: d_n and dd_nt (halved)
    V dm[3], sm[3], dX[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        dm[k] = b.m[k] - a.m[k];
        sm[k] = b.m[k] + a.m[k];
        dX[k] = vfma(b.m[k], c.B[1], zero - a.m[k] * c.A[1]);  // of m_a u_n
    }
    const V sX = vfma(b.m[0], c.B[1], a.m[0] * c.A[1]);
    const V de = b.e - a.e, se = b.e + a.e;
    const V dmt = vfma(b.m[0], c.B[4], zero - a.m[0] * c.A[4]);  // of m_n tau
    const V dln1 = b.ln1 - a.ln1, dl11 = b.l11 - a.l11;
    const V dln2 = b.ln2 - a.ln2, dl22 = b.l22 - a.l22;
    const V dodd = (b.o1 - a.o1) + (b.o2 - a.o2);
    const V dd = c.B[0] - c.A[0], sd = c.B[0] + c.A[0];  // of drho

    // the middle column
    const V* O = c.M;
    const V r = one + O[0];
    V m[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) m[k] = vfma(O[0], O[1 + k], O[1 + k]);
    V X0[3];  // m_a u_n
#pragma unroll
    for (int k = 0; k < 3; ++k) X0[k] = m[k] * O[1];
    const V e0 = vfma(O[0], Tbar + O[4], O[4]), mt0 = m[0] * O[4];
    // per tangent t = t1, t2 (S its slopes, u_t = O[2 + t]): the linear and
    // quadratic coefficients of m_a, the odd parts of m_a u_t and m_t tau,
    // the quadratic coefficients of m_t u_t and e
    V l[2][3], q[2][3], odd[2][3], mto[2], Xq[2], eq[2];
#pragma unroll
    for (int t = 0; t < 2; ++t) {
        const V* S = t == 0 ? c.M1 : c.M2;
        const V st = S[2 + t], ut = O[2 + t];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            l[t][k] = vfma(r, S[1 + k], S[0] * O[1 + k]);
            q[t][k] = S[0] * S[1 + k];
            const V mq = m[k] + q[t][k];
            odd[t][k] = vfma(st, mq, l[t][k] * ut);
            if (k == 1 + t) mto[t] = vfma(S[4], mq, l[t][k] * O[4]);
        }
        Xq[t] = vfma(l[t][1 + t], st, q[t][1 + t] * ut);
        eq[t] = S[0] * S[4];
    }
    // t1 t2 coefficients of m_1, m_2 and m_1 u_2
    const V k1 = vfma(c.M1[0], c.M2[2], c.M2[0] * c.M1[2]);
    const V k2 = vfma(c.M1[0], c.M2[3], c.M2[0] * c.M1[3]);
    const V k12 = vfma(l[0][1], c.M2[3], vfma(l[1][1], c.M1[3], k1 * O[3]));
    const V lt = l[0][1] + l[1][2];  // 1/2 (d_t1 m_1 + d_t2 m_2)
    const V hdiv = vfma(half, dm[0], lt);  // 1/2 sum_a d_a m_a

    // Eq. 46: drho*
    V drs = (O[0] - hdiv) + ((Xq[0] + Xq[1]) + k12);
    drs = vfma(half, vfma(m2, X0[0], sX) + dodd, drs);
    drs = vfma(hcs2, vfma(m2, O[0], sd), drs);
    // Eq. 47: m_a*
    V ms[3];
    {
        const V br = vfma(two, q[0][0] + q[1][0], dl11 + dl22);
        ms[0] = vfma(hcs2, vfma(three, vfma(m2, m[0], sm[0]), br),
                     vfma(mhalf, vfma(cs2, dd, dX[0]), m[0] - (odd[0][0] + odd[1][0])));
    }
    {
        const V br = vfma(two, q[1][1] + k2, dln1 + vfma(m2, m[1], sm[1]));
        ms[1] = vfma(hcs2, vfma(six, q[0][1], br),
                     vfma(mhalf, dX[1], vfma(mcs2, c.M1[0], m[1] - (odd[0][1] + odd[1][1]))));
    }
    {
        const V br = vfma(two, q[0][2] + k1, dln2 + vfma(m2, m[2], sm[2]));
        ms[2] = vfma(hcs2, vfma(six, q[1][2], br),
                     vfma(mhalf, dX[2], vfma(mcs2, c.M2[0], m[2] - (odd[0][2] + odd[1][2]))));
    }
    // Eq. 48: e* = (rho T)* - Tbar
    V es = (e0 - (mto[0] + mto[1])) - Tbar * hdiv;
    es = vfma(mhalf, dmt, es);
    es = vfma(hcs2, vfma(two, eq[0] + eq[1], vfma(m2, e0, se)), es);

    const V rho_s = one + drs;
    wall(ms[0], ms[1], ms[2], rho_s);
    const V inv = T::rcp(rho_s);
    const V un_s = ms[0] * inv;
    const V taus = (es - drs * Tbar) * inv;  // T* - Tbar

    // Eqs. 57-59 braces along +n
    F[0] = ms[0];
    {
        // a = n: X_nn = m_n u_n + cs2 drho, viscous 3 d_n m_n + d_t1 m_t1 + d_t2 m_t2
        const V Xn = vfma(cs2, O[0], X0[0]);
        F[1] = vfma(fl.m_nu_2h, vfma(three, dm[0], two * lt),
                    vfma(fl.m_tf15, vfma(ms[0], un_s, cs2 * drs) - Xn, Xn));
    }
#pragma unroll
    for (int k = 1; k < 3; ++k)
        F[1 + k] = vfma(fl.m_nu_2h, vfma(two, l[k - 1][0], dm[k]),
                        vfma(fl.m_tf15, vfma(ms[k], un_s, zero - X0[k]), X0[k]));
    {
        // (rho u_n T)* - (rho u_n T)^n = Tbar (m_n* - m_n) + m_n* tau* - m_n tau
        const V Q0 = vfma(m[0], Tbar, mt0);
        const V dQ = vfma(Tbar, ms[0] - m[0], vfma(ms[0], taus, zero - mt0));
        F[4] = vfma(fl.m_chi_2h, de, vfma(fl.m_tg15, dQ, Q0));
    }
}

template <typename V>
__host__ __device__ __forceinline__ void face_flux3(const CellNT3<V>& L, const CellNT3<V>& Rc,
                                                   V Tbar, const FaceLine<V>& fl, V keep, V uw1,
                                                   V uw2, V F[5])
{
    Cols3<V> c;
    face3_columns<V>(L, Rc, fl, c);
    // wall faces: no mass through the wall, the wall's tangential velocity
    face_flux3_wall<V>(c, Tbar, fl,
                       [&](V& mn, V& m1, V& m2, V rho) {
                           mn = mn * keep;
                           m1 = vfma(keep, m1, rho * uw1);
                           m2 = vfma(keep, m2, rho * uw2);
                       },
                       F);
}

// The original TLBFS face stage (Section 2.2) with D3Q19, from the same
// inputs and in the same frame as face_flux3: (a) equilibria (Eqs. 3-4,
// c_p = 1) at the nodes x_S - e_i h, i.e. node -e_i of the column form
// (Eq. 29); (b) the predicted variables as their moments (Eqs. 30-32), then
// the wall rule; (c) the fluxes of Eqs. 38-40 from the equilibria of the
// predicted variables and the non-equilibrium parts of Eqs. 33-34.
// Equilibria are carried as deviations f_i - w_i and g_i - w_i Tbar; the
// constants cancel in every moment used except the pressure c_s^2 of the
// normal momentum flux, which is dropped as in face_flux3.
//
// The moments of the predicted state's equilibria that a flux needs are
// exact (c_s^2 rho + rho u_n u_n, rho u_n u_t, rho u_n T), so only the
// nodes' equilibria are formed one by one, without their weights, and summed
// by weight and sign (as in the 2D stage).
template <typename V, class W>
__host__ __device__ __forceinline__ void face_flux3_tlbfs_wall(const CellNT3<V>& L,
                                                              const CellNT3<V>& Rc, V Tbar,
                                                              const FaceLine<V>& fl, W wall, V F[5])
{
    using T = vtraits<V>;
    const V one = T::bc(1.0), c45 = T::bc(4.5), mc15 = T::bc(-1.5), cs2 = T::bc(1.0 / 3.0);
    const V w0 = T::bc(1.0 / 3.0), w1 = T::bc(1.0 / 18.0), w2 = T::bc(1.0 / 36.0);
    const V half = T::bc(0.5), h = fl.h;
    const V wL = fl.cL + h, mwR = fl.cR - h;
    // columns a = -1 (left plane), 0 (mean), +1 (right plane): value + slopes in t1, t2
    V C[3][5], S1[3][5], S2[3][5];
#pragma unroll
    for (int k = 0; k < 5; ++k) {
        C[0][k] = vfma(L.gn[k], fl.cL, L.q[k]);
        S1[0][k] = L.g1[k] * h;
        S2[0][k] = L.g2[k] * h;
        C[2][k] = vfma(Rc.gn[k], fl.cR, Rc.q[k]);
        S1[2][k] = Rc.g1[k] * h;
        S2[2][k] = Rc.g2[k] * h;
        C[1][k] = half * (vfma(L.gn[k], wL, L.q[k]) + vfma(Rc.gn[k], mwR, Rc.q[k]));
        S1[1][k] = half * (S1[0][k] + S1[2][k]);
        S2[1][k] = half * (S2[0][k] + S2[2][k]);
    }
    // equilibria of direction (en, e1, e2) at the node opposite, over their
    // weights: f_i / w_i - 1 = drho + rho (3 eu + 4.5 eu^2 - 1.5 u^2), and
    // g_i / w_i - Tbar
    auto equil = [&](int en, int e1, int e2, V& f, V& g) {
        const int a = 1 - en;
        V q[5];
#pragma unroll
        for (int k = 0; k < 5; ++k) {
            V x = C[a][k];
            if (e1 < 0) x = x + S1[a][k];
            if (e1 > 0) x = x - S1[a][k];
            if (e2 < 0) x = x + S2[a][k];
            if (e2 > 0) x = x - S2[a][k];
            q[k] = x;
        }
        const V e = vfma(q[0], Tbar + q[4], q[4]);
        const V u2 = mc15 * vfma(q[1], q[1], vfma(q[2], q[2], q[3] * q[3]));
        if (en == 0 && e1 == 0 && e2 == 0) {
            f = vfma(one + q[0], u2, q[0]);
            g = e;
            return;
        }
        // eu = sign * s, s one velocity or the sum or difference of two
        const int sg = en != 0 ? en : (e1 != 0 ? e1 : e2);
        V s = en != 0 ? q[1] : (e1 != 0 ? q[2] : q[3]);
        if (en != 0 && e1 != 0) s = en == e1 ? s + q[2] : s - q[2];
        if ((en != 0 || e1 != 0) && e2 != 0) s = sg == e2 ? s + q[3] : s - q[3];
        const V three = T::bc(sg > 0 ? 3.0 : -3.0);
        f = vfma(one + q[0], vfma(s, vfma(c45, s, three), u2), q[0]);
        g = vfma(three * s, Tbar + e, e);
    };
    // opposite directions together: sum and difference of f and g
    auto both = [&](int en, int e1, int e2, V& sf, V& df, V& sg, V& dg) {
        V fp, gp, fm, gm;
        equil(en, e1, e2, fp, gp);
        equil(-en, -e1, -e2, fm, gm);
        sf = fp + fm;
        df = fp - fm;
        sg = gp + gm;
        dg = gp - gm;
    };
    // the predicted variables as moments, with those of the fluxes
    V f0, g0, sf, df, sg, dg;
    equil(0, 0, 0, f0, g0);
    V An, Dn, Gn, En;  // axis directions, normal
    both(1, 0, 0, An, Dn, Gn, En);
    V S1s = An, G1s = Gn;
    V D1, D2;
    both(0, 1, 0, sf, D1, sg, dg);
    S1s = S1s + sf;
    G1s = G1s + sg;
    both(0, 0, 1, sf, D2, sg, dg);
    S1s = S1s + sf;
    G1s = G1s + sg;
    // edge directions: d1 = (n, t1), d2 = (n, t2), d3 = (t1, t2)
    V sa, da, ga, ea, sb, db, gb, eb;
    both(1, 1, 0, sa, da, ga, ea);
    both(1, -1, 0, sb, db, gb, eb);
    V Sn2 = sa + sb, G2s = ga + gb, mn2 = da + db, m12 = da - db, En2 = ea + eb;
    const V Xn1e = sa - sb;
    both(1, 0, 1, sa, da, ga, ea);
    both(1, 0, -1, sb, db, gb, eb);
    Sn2 = Sn2 + (sa + sb);
    G2s = G2s + (ga + gb);
    mn2 = mn2 + (da + db);
    V m22 = da - db;
    En2 = En2 + (ea + eb);
    const V Xn2e = sa - sb;
    both(0, 1, 1, sa, da, ga, ea);
    both(0, 1, -1, sb, db, gb, eb);
    const V S2s = Sn2 + (sa + sb);
    G2s = G2s + (ga + gb);
    m12 = m12 + (da + db);
    m22 = m22 + (da - db);
    const V drs = vfma(w0, f0, vfma(w1, S1s, w2 * S2s));
    const V es = vfma(w0, g0, vfma(w1, G1s, w2 * G2s));
    V mn = vfma(w1, Dn, w2 * mn2), m1 = vfma(w1, D1, w2 * m12), m2 = vfma(w1, D2, w2 * m22);
    const V Xnn = vfma(w1, An, w2 * Sn2), Xn1 = w2 * Xn1e, Xn2 = w2 * Xn2e;
    const V Qn = vfma(w1, En, w2 * En2);
    const V rho_s = one + drs;
    wall(mn, m1, m2, rho_s);
    const V un = mn * T::rcp(rho_s);
    // fluxes along +n: the moments of the predicted equilibria plus the
    // non-equilibrium parts; 1/2 - tau = -3 nu / h = 6 (-nu / 2h) (Eqs. 9-10)
    const V cf = T::bc(6.0) * fl.m_nu_2h, cg = T::bc(6.0) * fl.m_chi_2h;
    const V Fnn = vfma(mn, un, cs2 * drs), Fn1 = m1 * un, Fn2 = m2 * un, Q = un * (Tbar + es);
    F[0] = mn;
    F[1] = vfma(cf, Fnn - Xnn, Fnn);
    F[2] = vfma(cf, Fn1 - Xn1, Fn1);
    F[3] = vfma(cf, Fn2 - Xn2, Fn2);
    F[4] = vfma(cg, Q - Qn, Q);
}

template <typename V>
__host__ __device__ __forceinline__ void face_flux3_tlbfs(const CellNT3<V>& L, const CellNT3<V>& Rc,
                                                         V Tbar, const FaceLine<V>& fl, V keep,
                                                         V uw1, V uw2, V F[5])
{
    face_flux3_tlbfs_wall<V>(L, Rc, Tbar, fl,
                             [&](V& mn, V& m1, V& m2, V rho) {
                                 mn = mn * keep;
                                 m1 = vfma(keep, m1, rho * uw1);
                                 m2 = vfma(keep, m2, rho * uw2);
                             },
                             F);
}

}  // namespace rtlbfs3
