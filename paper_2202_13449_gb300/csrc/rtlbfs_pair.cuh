// rtlbfs_pair.cuh -- two adjacent columns at once in packed FP32x2
// arithmetic: what the FP32 marching kernel (rtlbfs_march2.cu) and the FP32
// tile (rtlbfs_tile_pair.cuh) share.  A value of type f2 holds a quantity of
// columns a (x) and b = a + 1 (y).
#pragma once

#include <cuda_runtime.h>

#include "rtlbfs_dev.cuh"

namespace rtlbfs {

using Rec = Vec4<int>;  // a stored cell: (rho - 1, u, v, T) in fixed point

__device__ __forceinline__ f2 splat(float v) { return {v, v}; }

// two adjacent records at a 32-byte boundary in one access
__device__ __forceinline__ void ld2(const Rec* p, Rec& a, Rec& b)
{
    asm volatile("ld.global.v8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(a.x), "=r"(a.y), "=r"(a.z), "=r"(a.w), "=r"(b.x), "=r"(b.y), "=r"(b.z),
                   "=r"(b.w)
                 : "l"(p));
}
__device__ __forceinline__ void st2(Rec* p, const Rec& a, const Rec& b)
{
    asm volatile("st.global.v8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"l"(p), "r"(a.x), "r"(a.y),
                 "r"(a.z), "r"(a.w), "r"(b.x), "r"(b.y), "r"(b.z), "r"(b.w));
}

// A column's source on a line of n cells: the cell itself, the opposite
// cell of a periodic line, or the cell that a ghost up to two beyond a wall
// mirrors (m1, then m2: the sides to mirror across, -1: none).  Columns that
// no stencil uses give false.  With ghosts mirrored two deep the Green-Gauss
// gradient of the ghost column is the mirror of its partner's.
__device__ __forceinline__ bool column_source(int c, int n, bool per, int& src, int& m1, int& m2)
{
    const bool lo = c < 0, hi = c >= n;
    m2 = -1;
    if (per) {
        m1 = -1;
        src = lo ? c + n : (hi ? c - n : c);
        if ((unsigned)src >= (unsigned)n) src = ((c % n) + n) % n;  // a line shorter than a tile
        return true;
    }
    m1 = lo ? kSideW : (hi ? kSideE : -1);
    src = lo ? -1 - c : (hi ? 2 * n - 1 - c : c);
    if (c < -2 || c > n + 1) return false;
    if (n == 1 && (unsigned)src >= 1u) {  // the partner is itself a ghost
        m2 = m1;
        m1 = lo ? kSideE : kSideW;
        src = 0;
    }
    return true;
}

// A row's source: the row itself (halo rows of a strip are stored rows), the
// opposite row of a periodic side, or the row a ghost mirrors across side ym
// (-1: none).  Rows that no stencil uses give false.
__device__ __forceinline__ bool row_source(int r, int n, bool per, bool hlo, bool hhi, int& src,
                                           int& ym)
{
    ym = -1;
    src = r;
    if ((r >= 0 && r < n) || (r < 0 && hlo && r >= -2) || (r >= n && hhi && r <= n + 1)) return true;
    if (per) {
        src = r < 0 ? r + n : r - n;
        if ((unsigned)src >= (unsigned)n) src = ((r % n) + n) % n;
        return true;
    }
    if (r == -1) {
        src = 0;
        ym = kSideS;
        return true;
    }
    if (r == n) {
        src = n - 1;
        ym = kSideN;
        return true;
    }
    return false;
}

// Ghost values across wall `side` (-1: the values themselves) from the
// partner's working values (rho - 1, u, v, T - Tref): rho even, velocity odd
// about the wall velocity (normal component about 0), T odd about T_wall on
// a Dirichlet wall, even on an adiabatic one.  Selected without a branch:
// lanes across several sides would take it once for each.
__device__ __forceinline__ void mirror_values2(const CavityDesc& d, int side, float Tref, float v[4])
{
    const int k = max(side, 0);
    const float ut2 = 2.0f * d.f_bcU[k], T2 = 2.0f * (d.f_bcT[k] - Tref);
    const bool on = side >= 0, xn = k == kSideW || k == kSideE;
    v[1] = on ? (xn ? 0.0f : ut2) - v[1] : v[1];
    v[2] = on ? (xn ? ut2 : 0.0f) - v[2] : v[2];
    v[3] = on && d.kind[k] == kDirichlet ? T2 - v[3] : v[3];
}

// The ghost rules on a column's working values: row mirror first, then the
// column's (ok: a cell or ghost that some stencil uses; others are 0).
__device__ __forceinline__ void mirror_column(const CavityDesc& d, float Tref, bool ok, int ym,
                                              int m1, int m2, float v[4])
{
    mirror_values2(d, ym, Tref, v);
    mirror_values2(d, m1, Tref, v);
    if (m2 >= 0) mirror_values2(d, m2, Tref, v);
#pragma unroll
    for (int k = 0; k < 4; ++k) v[k] = ok ? v[k] : 0.0f;
}

// Gradient of a ghost row across a south or north wall: even quantities
// negate the normal part, odd ones the tangential part.
__device__ __forceinline__ void mirror_grad_rows(int kind, f2 gx[4], f2 gy[4])
{
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        if (wall_parity(kind, k) > 0) gy[k] = vtraits<f2>::neg(gy[k]);
        else gx[k] = vtraits<f2>::neg(gx[k]);
    }
}

// Working values (rho - 1, u, v, T - Tz) of two records.
__device__ __forceinline__ void convert2(const Rec& a, const Rec& b, int qTz, f2 v[4])
{
    const f2 x[4] = {{(float)a.x, (float)b.x},
                     {(float)a.y, (float)b.y},
                     {(float)a.z, (float)b.z},
                     {(float)(int)((unsigned)a.w - (unsigned)qTz),
                      (float)(int)((unsigned)b.w - (unsigned)qTz)}};
#pragma unroll
    for (int k = 0; k < 4; ++k) v[k] = x[k] * splat(StoreQ::scale_f(k));
}

// Fluxes of two faces with the same orientation from the cells on either
// side (working values v, gradients along x and y in storage order): F =
// (mass, x-, y-momentum, energy).  ISX: x-faces (normal u, tangential v).
// wall(mn, mt, rho): the wall rule on the predicted momenta.
template <bool ISX, int SCHEME, class W>
__device__ __forceinline__ void faces2(const f2 vl[4], const f2 gxl[4], const f2 gyl[4],
                                       const f2 vr[4], const f2 gxr[4], const f2 gyr[4], f2 Tz,
                                       const FaceLine<f2>& fl, W wall, f2 F[4])
{
    constexpr int N = ISX ? 1 : 2, S = ISX ? 2 : 1;
    constexpr int q[4] = {0, N, S, 3};
    const f2* nl = ISX ? gxl : gyl;
    const f2* tl = ISX ? gyl : gxl;
    const f2* nr = ISX ? gxr : gyr;
    const f2* tr = ISX ? gyr : gxr;
    CellNT<f2> L, R;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        L.q[k] = vl[q[k]];
        R.q[k] = vr[q[k]];
        L.gn[k] = nl[q[k]];
        R.gn[k] = nr[q[k]];
        L.gt[k] = tl[q[k]];
        R.gt[k] = tr[q[k]];
    }
    // temperatures relative to the left cell's (its own deviation is 0)
    const f2 Tbar = Tz + L.q[3];
    f2 G[4];
    R.q[3] = R.q[3] - L.q[3];
    L.q[3] = splat(0.0f);
    if constexpr (SCHEME == 1) {
        face_flux_tlbfs_wall<f2>(L, R, Tbar, fl, wall, G);
    } else {
        f2 A[4], Na[4], M[4], D[4], B[4], Sb[4];
        face_columns<f2>(L, R, fl, A, Na, M, D, B, Sb);
        face_flux_wall<f2>(A, Na, M, D, B, Sb, Tbar, fl, wall, G);
    }
    F[0] = G[0];
    F[N] = G[1];
    F[S] = G[2];
    F[3] = G[3];
}

// A face line's constants for a pair of faces that share it.
__device__ __forceinline__ FaceLine<f2> splat_line(const FaceLine<float>& p)
{
    FaceLine<f2> f;
    f.h = splat(p.h);
    f.cL = splat(p.cL);
    f.cR = splat(p.cR);
    f.m_nu_2h = splat(p.m_nu_2h);
    f.m_chi_2h = splat(p.m_chi_2h);
    f.m_tf15 = splat(p.m_tf15);
    f.m_tg15 = splat(p.m_tg15);
    f.pad = splat(0.0f);
    return f;
}

// Sums of a step's residual over pairs of cells.
struct PairSums {
    f2 s[4] = {{0.0f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}};
    bool bad = false;
};

// The warp's sums: lane l holds sum l / 8.
__device__ __forceinline__ float warp_total(const PairSums& a)
{
    return warp_sum4(a.bad ? NAN : a.s[0].x + a.s[0].y, a.s[1].x + a.s[1].y, a.s[2].x + a.s[2].y,
                     a.s[3].x + a.s[3].y);
}

// The explicit update of two cells (increment form) with the Boussinesq
// source (Eq. 64), from their working values v, the flux balance div (Dt/dV
// sum_k F_k dS_k) and the stored records qa, qb; the second cell counts only
// if both.  sfx, sfy, sbg: body force and buoyancy times the time step.
__device__ __forceinline__ void update2(const f2 v[4], float Tz, const f2 div[4], float sfx,
                                        float sfy, float sbg, float Tr, const Rec& qa, const Rec& qb,
                                        bool both, Rec* out, PairSums& acc)
{
    using P = StoreQ;
    const f2 dr = v[0], u = v[1], w = v[2], T = splat(Tz) + v[3];
    const f2 rho = splat(1.0f) + dr;
    const f2 src_x = rho * splat(sfx);
    const f2 src_y = rho * vfma(splat(sbg), T - splat(Tr), splat(sfy));
    // rho^{n+1} = rho - div0; q^{n+1} - q = (q div0 - div_q + dt src) / rho^{n+1}
    const f2 inv = vtraits<f2>::rcp(rho - div[0]);
    const f2 du = (vfma(u, div[0], src_x) - div[1]) * inv;
    const f2 dw = (vfma(w, div[0], src_y) - div[2]) * inv;
    const f2 dT = (T * div[0] - div[3]) * inv;
    const f2 dr1 = dr - div[0], u1 = u + du, w1 = w + dw, T1 = T + dT;
    const Rec oa = {P::add(qa.x, -div[0].x, 0), P::add(qa.y, du.x, 1), P::add(qa.z, dw.x, 2),
                    P::add(qa.w, dT.x, 3)};
    const Rec ob = {P::add(qb.x, -div[0].y, 0), P::add(qb.y, du.y, 1), P::add(qb.z, dw.y, 2),
                    P::add(qb.w, dT.y, 3)};
    const bool ba = !(P::in_range(dr1.x, 0) && P::in_range(u1.x, 1) && P::in_range(w1.x, 2) &&
                      P::in_range(T1.x, 3));
    const bool bb = !(P::in_range(dr1.y, 0) && P::in_range(u1.y, 1) && P::in_range(w1.y, 2) &&
                      P::in_range(T1.y, 3));
    // |u|^{n+1} - |u|^n without cancellation
    const f2 q0 = vfma(u, u, w * w), q1 = vfma(u1, u1, w1 * w1);
    const f2 den = f2{P::fsqrt(q0.x), P::fsqrt(q0.y)} + f2{P::fsqrt(q1.x), P::fsqrt(q1.y)};
    const f2 num = vfma(du, u + u1, dw * (w + w1));
    f2 dm = {den.x > 0.0f ? num.x * P::rcp(den.x) : 0.0f,
             den.y > 0.0f ? num.y * P::rcp(den.y) : 0.0f};
    f2 e1 = q1, e2 = dT, e3 = T1;
    acc.bad = acc.bad || ba || (bb && both);
    if (both) {
        st2(out, oa, ob);
    } else {  // the last column of an odd line: b is not a cell
        *out = oa;
        dm.y = e1.y = e2.y = e3.y = 0.0f;
    }
    acc.s[0] = vfma(dm, dm, acc.s[0]);
    acc.s[1] = acc.s[1] + e1;
    acc.s[2] = vfma(e2, e2, acc.s[2]);
    acc.s[3] = vfma(e3, e3, acc.s[3]);
}

}  // namespace rtlbfs
