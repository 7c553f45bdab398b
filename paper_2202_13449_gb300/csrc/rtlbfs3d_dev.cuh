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
// the same numbers with a third fewer operations (280 a face against 435
// for products at the 19 nodes), and without the cancellation of the node
// differences.  FP64 runs at the FMA rate, so there the step follows the
// count: 20 steps of an 80^3 mesh and the download, FP64, 34.8 -> 29.5 ms;
// FP32, bound by its shared-memory phases, is unchanged (21.8 ms for 300).
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

template <typename V>
__host__ __device__ __forceinline__ void face_flux3_columns(const Cols3<V>& c, V Tbar,
                                                           const FaceLine<V>& fl, V keep, V uw1,
                                                           V uw2, V F[5])
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
    // wall faces: no mass through the wall, the wall's tangential velocity
    ms[0] = ms[0] * keep;
    ms[1] = vfma(keep, ms[1], rho_s * uw1);
    ms[2] = vfma(keep, ms[2], rho_s * uw2);
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
    face_flux3_columns<V>(c, Tbar, fl, keep, uw1, uw2, F);
}

// face3_columns in FP32, components (0, 1) and (2, 3) in packed FP32x2 pairs
// (component 4 alone): the same operations, bit for bit.
__device__ __forceinline__ void face3_columns_f32(const CellNT3<float>& L, const CellNT3<float>& Rc,
                                                  const FaceLine<float>& fl, Cols3<float>& c)
{
    const float h = fl.h;
    const float wL = fl.cL + h, mwR = fl.cR - h, hh = h * 0.5f;
    const float2 cL2 = make_float2(fl.cL, fl.cL), cR2 = make_float2(fl.cR, fl.cR);
    const float2 wL2 = make_float2(wL, wL), mwR2 = make_float2(mwR, mwR);
    const float2 h2 = make_float2(h, h), hh2 = make_float2(hh, hh);
    const float2 half2 = make_float2(0.5f, 0.5f);
    auto pr = [](const float* a, int i) { return make_float2(a[2 * i], a[2 * i + 1]); };
    auto put = [](float* d, int i, float2 v) {
        d[2 * i] = v.x;
        d[2 * i + 1] = v.y;
    };
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const float2 q = pr(L.q, i), gn = pr(L.gn, i), g1 = pr(L.g1, i), g2 = pr(L.g2, i);
        const float2 qr = pr(Rc.q, i), gnr = pr(Rc.gn, i), g1r = pr(Rc.g1, i), g2r = pr(Rc.g2, i);
        put(c.A, i, __ffma2_rn(gn, cL2, q));
        put(c.A1, i, __fmul2_rn(g1, h2));
        put(c.A2, i, __fmul2_rn(g2, h2));
        put(c.B, i, __ffma2_rn(gnr, cR2, qr));
        put(c.B1, i, __fmul2_rn(g1r, h2));
        put(c.B2, i, __fmul2_rn(g2r, h2));
        put(c.M, i, __fmul2_rn(half2, __fadd2_rn(__ffma2_rn(gn, wL2, q), __ffma2_rn(gnr, mwR2, qr))));
        put(c.M1, i, __fmul2_rn(hh2, __fadd2_rn(g1, g1r)));
        put(c.M2, i, __fmul2_rn(hh2, __fadd2_rn(g2, g2r)));
    }
    c.A[4] = fmaf(L.gn[4], fl.cL, L.q[4]);
    c.B[4] = fmaf(Rc.gn[4], fl.cR, Rc.q[4]);
    c.M[4] = 0.5f * (fmaf(L.gn[4], wL, L.q[4]) + fmaf(Rc.gn[4], mwR, Rc.q[4]));
    c.M1[4] = hh * (L.g1[4] + Rc.g1[4]);
    c.M2[4] = hh * (L.g2[4] + Rc.g2[4]);
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
template <typename V>
__host__ __device__ __forceinline__ void face_flux3_tlbfs(const CellNT3<V>& L, const CellNT3<V>& Rc,
                                                         V Tbar, const FaceLine<V>& fl, V keep,
                                                         V uw1, V uw2, V F[5])
{
    using T = vtraits<V>;
    const V zero = T::bc(0.0), half = T::bc(0.5), one = T::bc(1.0), three = T::bc(3.0);
    const V c45 = T::bc(4.5), mc15 = T::bc(-1.5), six = T::bc(6.0);
    // D3Q19 (Eq. 5) in the face frame: the set is the same in every frame
    constexpr int en[19] = {0, 1, -1, 0, 0, 0, 0, 1, -1, 1, -1, 1, -1, 1, -1, 0, 0, 0, 0};
    constexpr int e1[19] = {0, 0, 0, 1, -1, 0, 0, 1, 1, -1, -1, 0, 0, 0, 0, 1, -1, 1, -1};
    constexpr int e2[19] = {0, 0, 0, 0, 0, 1, -1, 0, 0, 0, 0, 1, 1, -1, -1, 1, 1, -1, -1};
    const V w0 = T::bc(1.0 / 3.0), w1 = T::bc(1.0 / 18.0), w2 = T::bc(1.0 / 36.0);
    const V h = fl.h;
    const V wL = fl.cL + h, mwR = fl.cR - h;
    const V hh = h * half;
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
        S1[1][k] = hh * (L.g1[k] + Rc.g1[k]);
        S2[1][k] = hh * (L.g2[k] + Rc.g2[k]);
    }
    // (a), (b): equilibria at the nodes -e_i and their moments
    V df[19], dg[19];
    V drs = zero, mn = zero, m1 = zero, m2 = zero, es = zero;
#pragma unroll
    for (int i = 0; i < 19; ++i) {
        const int a = 1 - en[i], b = -e1[i], c = -e2[i];  // column, offsets along t1, t2
        V q[5];
#pragma unroll
        for (int k = 0; k < 5; ++k) {
            V x = C[a][k];
            if (b > 0) x = x + S1[a][k];
            if (b < 0) x = x - S1[a][k];
            if (c > 0) x = x + S2[a][k];
            if (c < 0) x = x - S2[a][k];
            q[k] = x;
        }
        const V w = i == 0 ? w0 : (i < 7 ? w1 : w2);
        V eu = zero;
        if (en[i] > 0) eu = eu + q[1];
        if (en[i] < 0) eu = eu - q[1];
        if (e1[i] > 0) eu = eu + q[2];
        if (e1[i] < 0) eu = eu - q[2];
        if (e2[i] > 0) eu = eu + q[3];
        if (e2[i] < 0) eu = eu - q[3];
        const V usq = vfma(q[1], q[1], vfma(q[2], q[2], q[3] * q[3]));
        const V rho = one + q[0];
        // f_i - w_i = w_i (drho + rho (3 eu + 4.5 eu^2 - 1.5 u^2))
        df[i] = w * vfma(rho, vfma(eu, vfma(c45, eu, three), mc15 * usq), q[0]);
        // rho T - Tbar at the node, and g_i - w_i Tbar
        const V e_node = vfma(q[0], Tbar + q[4], q[4]);
        dg[i] = w * vfma(three * eu, Tbar + e_node, e_node);
        drs = drs + df[i];
        if (en[i] > 0) mn = mn + df[i];
        if (en[i] < 0) mn = mn - df[i];
        if (e1[i] > 0) m1 = m1 + df[i];
        if (e1[i] < 0) m1 = m1 - df[i];
        if (e2[i] > 0) m2 = m2 + df[i];
        if (e2[i] < 0) m2 = m2 - df[i];
        es = es + dg[i];
    }
    const V rho_s = one + drs;
    mn = mn * keep;
    const V wallr = (one - keep) * rho_s;
    m1 = vfma(keep, m1, wallr * uw1);
    m2 = vfma(keep, m2, wallr * uw2);
    const V inv = T::rcp(rho_s);
    const V un = mn * inv, u1 = m1 * inv, u2 = m2 * inv;
    const V usq_s = vfma(un, un, vfma(u1, u1, u2 * u2));
    // (c) fluxes along +n; 1/2 - tau = -3 nu / h = 6 (-nu / 2h) (Eqs. 9-10)
    const V cf = six * fl.m_nu_2h, cg = six * fl.m_chi_2h;
    V Fnn = zero, Fn1 = zero, Fn2 = zero, Q = zero;
#pragma unroll
    for (int i = 0; i < 19; ++i) {
        if (en[i] == 0) continue;  // no flux along n
        const V w = i < 7 ? w1 : w2;
        V eu = en[i] > 0 ? un : zero - un;
        if (e1[i] > 0) eu = eu + u1;
        if (e1[i] < 0) eu = eu - u1;
        if (e2[i] > 0) eu = eu + u2;
        if (e2[i] < 0) eu = eu - u2;
        const V dfs = w * vfma(rho_s, vfma(eu, vfma(c45, eu, three), mc15 * usq_s), drs);
        const V dgs = w * vfma(three * eu, Tbar + es, es);
        const V pf = vfma(cf, dfs - df[i], dfs);  // f* + (1/2 - tau_f)(f* - f_node)
        const V pg = vfma(cg, dgs - dg[i], dgs);
        Fnn = Fnn + pf;  // e_n^2 = 1
        if (e1[i] != 0) Fn1 = (en[i] * e1[i] > 0) ? Fn1 + pf : Fn1 - pf;
        if (e2[i] != 0) Fn2 = (en[i] * e2[i] > 0) ? Fn2 + pf : Fn2 - pf;
        Q = en[i] > 0 ? Q + pg : Q - pg;
    }
    F[0] = mn;
    F[1] = Fnn;
    F[2] = Fn1;
    F[3] = Fn2;
    F[4] = Q;
}

}  // namespace rtlbfs3
