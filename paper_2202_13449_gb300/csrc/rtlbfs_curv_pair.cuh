// rtlbfs_curv_pair.cuh -- the FP32 curvilinear step in packed pairs of cells
// adjacent along i (included by rtlbfs_curv.cu; FP64: curv_step_kernel there).
//
// The phases of curv_step_kernel on the same tiles, one thread per pair of
// cells.  A thread per cell in scalar arithmetic, with the geometry as records,
// ran 1980 instructions a cell; this runs 1000 (its share of the copies, loads
// and ghost items included).  Steps of 300 x 200, 450 x 300 and 1800 x 1200
// cells: 6.6, 9.1 and 120 us, before 8.35, 11.4 and 161.
// Small meshes are bound by the chain of latencies from one launch to the
// next (5.6 us at 150 x 100), large ones by how many warps the 46 KB of staged
// geometry per block let wait for shared memory: 2.8 TB/s and half of the
// issue slots at 1800 x 1200.
//
// Ghost columns hold values mirrored two deep and carry Green-Gauss
// coefficients of their own (see pair_geo), so their gradients need no rule;
// a ghost row takes its partner row's differences with reflected
// coefficients and the sign of the quantity.
#pragma once

namespace rtlbfsc {

using rtlbfs::f2;
using rtlbfs::splat;
using rtlbfs::vtraits;

// Geometry rows of a strip of kPairX columns, as the kernel stages them: per
// row, one field after another over the columns, so that a tile's rows are
// contiguous and a pair of columns is one 8-byte access.
constexpr int kPairX = 32;
struct PairRow {
    float c[8][kPairX + 4];  // CellGrad of columns -2 .. kPairX + 1 (rows -1 .. nj)
};
struct PairFaceI {
    float f[12][kPairX + 2];  // FaceRec fields of the i-faces 0 .. kPairX (rows 0 .. nj - 1)
};
struct PairFaceJ {
    float f[12][kPairX];  // FaceRec fields of the j-faces (rows 0 .. nj)
};
enum { kNx, kNy, kTL, kTR, kH, kCL, kCR, kNu2h, kChi2h, kTf15, kTg15, kLen };

template <int TY>
struct SmemCP {
    static constexpr int PX = kPairX / 2, NP = PX + 2, BY = TY + 4, GY = TY + 2, NT = PX * TY;
    PairRow g[GY];        // coefficients, overwritten by the gradients
    PairFaceJ fj[TY + 1];  // each face's flux is written over its fields 0 .. 3
    PairFaceI fi[TY];
    float dta[TY][kPairX];
    f2 v[4][BY][NP];
    float red[NT / 32][4];
    int plan[3];  // after the stop test: done, cur, sum slot
};

// Two faces with the cells' working values (rho - 1, u, v, T - Tz) and
// gradients g[2 q + axis]; geo: the faces' FaceRec fields.  wall(mn, mt,
// rho, tx, ty): the wall rule on the predicted momenta, tangent (tx, ty).
// Returns the fluxes times the face length in x, y components.
template <class W>
__device__ __forceinline__ void faces_c2(const f2 vL[4], const f2 gL[8], const f2 vR[4],
                                         const f2 gR[8], const f2 geo[12], f2 Tz, W wall, f2 out[4])
{
    const f2 nx = geo[kNx], ny = geo[kNy], tx = vtraits<f2>::neg(ny);
    rtlbfs::CellNT<f2> L, R;
    auto frame = [&](const f2 v[4], const f2 g[8], f2 mt, rtlbfs::CellNT<f2>& c) {
        auto rot_n = [&](f2 x, f2 y) { return vfma(nx, x, ny * y); };
        auto rot_t = [&](f2 x, f2 y) { return vfma(tx, x, nx * y); };
        const f2 gnu = rot_n(g[2], g[3]), gtu = rot_t(g[2], g[3]);
        const f2 gnv = rot_n(g[4], g[5]), gtv = rot_t(g[4], g[5]);
        c.gn[0] = rot_n(g[0], g[1]);
        c.gt[0] = rot_t(g[0], g[1]);
        c.gn[1] = rot_n(gnu, gnv);
        c.gt[1] = rot_n(gtu, gtv);
        c.gn[2] = rot_t(gnu, gnv);
        c.gt[2] = rot_t(gtu, gtv);
        c.gn[3] = rot_n(g[6], g[7]);
        c.gt[3] = rot_t(g[6], g[7]);
        // values on the face's normal line: the centre's tangential offset folded in
        c.q[0] = vfma(c.gt[0], mt, v[0]);
        c.q[1] = vfma(c.gt[1], mt, rot_n(v[1], v[2]));
        c.q[2] = vfma(c.gt[2], mt, rot_t(v[1], v[2]));
        c.q[3] = vfma(c.gt[3], mt, v[3]);
    };
    frame(vL, gL, vtraits<f2>::neg(geo[kTL]), L);
    frame(vR, gR, vtraits<f2>::neg(geo[kTR]), R);
    const f2 Tbar = Tz + L.q[3];
    R.q[3] = R.q[3] - L.q[3];
    L.q[3] = splat(0.0f);
    const FaceLine<f2> fl = {geo[kH],    geo[kCL],    geo[kCR],   geo[kNu2h],
                             geo[kChi2h], geo[kTf15], geo[kTg15], splat(0.0f)};
    f2 A[4], Na[4], M[4], D[4], B[4], Sb[4], F[4];
    rtlbfs::face_columns<f2>(L, R, fl, A, Na, M, D, B, Sb);
    rtlbfs::face_flux_wall<f2>(A, Na, M, D, B, Sb, Tbar, fl,
                               [&](f2& mn, f2& mt, f2 rho) { wall(mn, mt, rho, tx, nx); }, F);
    const f2 len = geo[kLen];
    out[0] = F[0] * len;
    out[1] = vfma(F[1], nx, F[2] * tx) * len;
    out[2] = vfma(F[1], ny, F[2] * nx) * len;
    out[3] = F[3] * len;
}

__device__ __forceinline__ f2 at2(const float* p) { return *reinterpret_cast<const f2*>(p); }
__device__ __forceinline__ void put2(float* p, f2 x) { *reinterpret_cast<f2*>(p) = x; }

// n 16-byte groups from a 16-byte aligned array
template <int NT>
__device__ __forceinline__ void stage16(void* dst, const void* src, int bytes)
{
    for (int t = threadIdx.x; t < bytes / 16; t += NT)
        cp_async16(static_cast<unsigned char*>(dst) + 16 * t,
                   static_cast<const unsigned char*>(src) + 16 * t);
}

template <int TY>
__global__ void __launch_bounds__(SmemCP<TY>::NT, 512 / SmemCP<TY>::NT)
curv_pair_kernel(const DescC* __restrict__ dp, CavityRun* __restrict__ run, int par)
{
    using P = StoreQ;
    using Sm = SmemCP<TY>;
    using Rec = Vec4<int>;
    constexpr int PX = Sm::PX, NP = Sm::NP, BY = Sm::BY, GY = Sm::GY, NT = Sm::NT;
    static_assert(sizeof(PairRow) % 16 == 0 && sizeof(PairFaceI) % 16 == 0, "staged in 16-byte groups");
    extern __shared__ __align__(16) unsigned char smraw[];
    Sm& sm = *reinterpret_cast<Sm*>(smraw);
    const DescC& d = *dp;
    const int tid = threadIdx.x, px = tid % PX, ty = tid / PX, lane = tid & 31, warp = tid >> 5;
    const int ni = d.ni, nj = d.nj, rows = d.pair_rows;
    const bool per = d.per != 0;
    // read ahead of the copies, one latency for all
    const PairRow* cg = static_cast<const PairRow*>(d.cg);
    const PairFaceI* fri = static_cast<const PairFaceI*>(d.fri);
    const PairFaceJ* frj = static_cast<const PairFaceJ*>(d.frj);
    const float* dta = static_cast<const float*>(d.dta);
    void *const rec0 = d.rec[0], *const rec1 = d.rec[1];
    const int strip = blockIdx.x % d.tiles_x;
    const int i0 = strip * kPairX, j0 = (blockIdx.x / d.tiles_x) * TY;

    // 0. the tile's geometry (constant across steps) into shared memory; the
    // strips are stored to a multiple of the tile height
    stage16<NT>(sm.g, cg + (size_t)strip * (rows + 2) + j0, sizeof(sm.g));
    stage16<NT>(sm.fj, frj + (size_t)strip * (rows + 1) + j0, sizeof(sm.fj));
    stage16<NT>(sm.fi, fri + (size_t)strip * rows + j0, sizeof(sm.fi));
    stage16<NT>(sm.dta, dta + ((size_t)strip * rows + j0) * kPairX, sizeof(sm.dta));
    cp_async_commit();

    chain_sync();
    // the stop test of the previous step (thread 0; unit 0 publishes the
    // header for the next launch)
    if (tid == 0) {
        const CavityCtl dc = rtlbfs::run_head(run, par);
        if (blockIdx.x == 0) rtlbfs::run_publish(run, par, dc);
        sm.plan[0] = dc.done;
        sm.plan[1] = dc.cur;
        sm.plan[2] = (int)(dc.steps % 3);
    }
    __syncthreads();
    if (sm.plan[0]) {  // uniform
        cp_async_wait_all();
        return;
    }
    const int cur = sm.plan[1], slot3 = sm.plan[2];
    const Rec* __restrict__ rin = static_cast<const Rec*>(cur ? rec1 : rec0);
    Rec* __restrict__ rout = static_cast<Rec*>(cur ? rec0 : rec1);
    const int qTz = rin[(size_t)min(j0 + TY / 2, nj - 1) * ni + min(i0 + kPairX / 2, ni - 1)].w;
    const float Tz = P::val(qTz, 3);
    const f2 Tz2 = splat(Tz);
    const int gi = i0 + 2 * px, gj = j0 + ty;
    const bool mine = gi < ni && gj < nj, both = gi + 1 < ni;
    const size_t off = (size_t)gj * ni + gi;

    // 1. values on the tile and a 2-cell ring: the row's ghost rule first,
    // then the column's
#pragma unroll
    for (int k = 0; k < (NP * BY + NT - 1) / NT; ++k) {
        const int t = tid + k * NT, r = t / NP, p = t - r * NP;
        if (t >= NP * BY) break;
        int js, ys;
        const bool row = resolve_c(j0 - 2 + r, nj, false, 2, 3, js, ys);
        int s[2], m1[2], m2[2];
        bool ok[2];
        Rec q[2];
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            ok[c] = rtlbfs::column_source(i0 - 2 + 2 * p + c, ni, per, s[c], m1[c], m2[c]) && row;
            q[c] = rin[ok[c] ? (size_t)js * ni + s[c] : 0];
        }
        f2 v[4];
        rtlbfs::convert2(q[0], q[1], qTz, v);
        if (!(ok[0] && ok[1]) || ys >= 0 || m1[0] >= 0 || m1[1] >= 0) {
            float w[2][4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                w[0][e] = v[e].x;
                w[1][e] = v[e].y;
            }
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                if (ys >= 0) ghost_values<P, float>(d, ys, Tz, w[c]);
                if (m1[c] >= 0) ghost_values<P, float>(d, m1[c], Tz, w[c]);
                if (m2[c] >= 0) ghost_values<P, float>(d, m2[c], Tz, w[c]);
            }
#pragma unroll
            for (int e = 0; e < 4; ++e) v[e] = {ok[0] ? w[0][e] : 0.0f, ok[1] ? w[1][e] : 0.0f};
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) sm.v[e][r][p] = v[e];
    }
    cp_async_wait_all();
    __syncthreads();

    // 2. gradients on the tile and a 1-cell ring
#pragma unroll 1
    for (int t = tid; t < NP * GY; t += NT) {
        const int gr = t / NP, p = t - gr * NP, j = j0 - 1 + gr;
        const int ys = j == -1 ? 2 : (j == nj ? 3 : -1);  // a ghost row
        const int r = gr + 1 + (ys == 2 ? 1 : (ys == 3 ? -1 : 0));
        // neighbours of the ring's outer columns are not read by any face
        const int wp = max(p - 1, 0), ep = min(p + 1, NP - 1);
        f2 c[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) c[e] = at2(&sm.g[gr].c[e][2 * p]);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const f2 o = sm.v[q][r][p];
            const f2 de = f2{o.y, sm.v[q][r][ep].x} - o, dw = f2{sm.v[q][r][wp].y, o.x} - o;
            const f2 dn = sm.v[q][r + 1][p] - o, ds = sm.v[q][r - 1][p] - o;
            f2 gx = vfma(c[0], de, vfma(c[2], dw, vfma(c[4], dn, c[6] * ds)));
            f2 gy = vfma(c[1], de, vfma(c[3], dw, vfma(c[5], dn, c[7] * ds)));
            if (ys >= 0 && (q == 1 || q == 2 || (q == 3 && d.kind[ys] == kDir))) {
                gx = vtraits<f2>::neg(gx);
                gy = vtraits<f2>::neg(gy);
            }
            put2(&sm.g[gr].c[2 * q][2 * p], gx);
            put2(&sm.g[gr].c[2 * q + 1][2 * p], gy);
        }
    }
    __syncthreads();

    // 3. faces of the tile; each face's flux replaces its record
    auto cell = [&](int r, int p, f2 v[4], f2 g[8]) {
#pragma unroll
        for (int q = 0; q < 4; ++q) v[q] = sm.v[q][r][p];
#pragma unroll
        for (int e = 0; e < 8; ++e) g[e] = at2(&sm.g[r - 1].c[e][2 * p]);
    };
#pragma unroll 1
    for (int it = 0; it < 2; ++it) {  // i-faces west of a and between a and b; the tile's east column
        const int row = it ? lane : ty, p = it ? PX : px;
        if (it && (warp != 0 || lane >= TY)) continue;
        f2 vL[4], gL[8], vR[4], gR[8], geo[12], F[4];
        cell(row + 2, p + 1, vR, gR);
        cell(row + 2, p, vL, gL);  // the pair to the west: its b, then a
#pragma unroll
        for (int q = 0; q < 4; ++q) vL[q] = {vL[q].y, vR[q].x};
#pragma unroll
        for (int e = 0; e < 8; ++e) gL[e] = {gL[e].y, gR[e].x};
#pragma unroll
        for (int e = 0; e < 12; ++e) geo[e] = at2(&sm.fi[row].f[e][2 * p]);
        const int g = i0 + 2 * p;
        faces_c2(vL, gL, vR, gR, geo, Tz2,
                 [&](f2& mn, f2& mt, f2 rho, f2 tx, f2 ty) {
                     if (per) return;
                     if ((g == 0 || g == ni) && d.kind[g == 0 ? 0 : 1] != kFar) {
                         const int s = g == 0 ? 0 : 1;
                         mn.x = 0.0f;
                         mt.x = rho.x * (d.f_bcU[s][0] * tx.x + d.f_bcU[s][1] * ty.x);
                     }
                     if (g + 1 == ni && d.kind[1] != kFar) {
                         mn.y = 0.0f;
                         mt.y = rho.y * (d.f_bcU[1][0] * tx.y + d.f_bcU[1][1] * ty.y);
                     }
                 },
                 F);
#pragma unroll
        for (int q = 0; q < 4; ++q) put2(&sm.fi[row].f[q][2 * p], F[q]);
    }
#pragma unroll 1
    for (int it = 0; it < 2; ++it) {  // j-faces south of a and b; the tile's north row
        const int row = it ? TY : ty, p = it ? lane : px;
        if (it && (warp != NT / 32 - 1 || lane >= PX)) continue;
        f2 vL[4], gL[8], vR[4], gR[8], geo[12], F[4];
        cell(row + 1, p + 1, vL, gL);
        cell(row + 2, p + 1, vR, gR);
#pragma unroll
        for (int e = 0; e < 12; ++e) geo[e] = at2(&sm.fj[row].f[e][2 * p]);
        const int g = j0 + row;
        faces_c2(vL, gL, vR, gR, geo, Tz2,
                 [&](f2& mn, f2& mt, f2 rho, f2 tx, f2 ty) {
                     const int s = g == 0 ? 2 : (g == nj ? 3 : -1);
                     if (s >= 0 && d.kind[s] != kFar) {
                         mn = splat(0.0f);
                         mt = rho * vfma(splat(d.f_bcU[s][0]), tx, splat(d.f_bcU[s][1]) * ty);
                     }
                 },
                 F);
#pragma unroll
        for (int q = 0; q < 4; ++q) put2(&sm.fj[row].f[q][2 * p], F[q]);
    }
    Rec qa = {0, 0, 0, 0}, qb = qa;
    if (mine) {  // the stored cells the update adds its increments to
        qa = rin[off];
        if (both) qb = rin[off + 1];
    }
    __syncthreads();

    // 4. update
    float s0 = 0.0f, s1 = 0.0f, s2 = 0.0f, s3 = 0.0f;
    bool bad = false;
    if (mine) {
        const f2 a = at2(&sm.dta[ty][2 * px]);
        f2 div[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const f2 w = at2(&sm.fi[ty].f[q][2 * px]);
            const f2 e = {w.y, sm.fi[ty].f[q][2 * px + 2]};
            div[q] = a * ((e - w) + (at2(&sm.fj[ty + 1].f[q][2 * px]) - at2(&sm.fj[ty].f[q][2 * px])));
        }
        const f2 dr = sm.v[0][ty + 2][px + 1], u = sm.v[1][ty + 2][px + 1];
        const f2 v = sm.v[2][ty + 2][px + 1], T = Tz2 + sm.v[3][ty + 2][px + 1];
        const f2 rho = splat(1.0f) + dr;
        const float dtc = d.f_dt;
        const f2 b = splat(d.f_beta_g) * (T - splat(d.f_T_ref));
        const f2 srcx = splat(dtc) * (rho * vfma(b, splat(d.f_gdir[0]), splat(d.f_force[0])));
        const f2 srcy = splat(dtc) * (rho * vfma(b, splat(d.f_gdir[1]), splat(d.f_force[1])));
        const f2 inv = vtraits<f2>::rcp(rho - div[0]);
        const f2 du = (vfma(u, div[0], srcx) - div[1]) * inv;
        const f2 dv = (vfma(v, div[0], srcy) - div[2]) * inv;
        const f2 dT = (T * div[0] - div[3]) * inv;
        const f2 dr1 = dr - div[0], u1 = u + du, v1 = v + dv, T1 = T + dT;
        rout[off] = {P::add(qa.x, -div[0].x, 0), P::add(qa.y, du.x, 1), P::add(qa.z, dv.x, 2),
                     P::add(qa.w, dT.x, 3)};
        bad = !(P::in_range(dr1.x, 0) && P::in_range(u1.x, 1) && P::in_range(v1.x, 2) &&
                P::in_range(T1.x, 3));
        const f2 q0 = vfma(u, u, v * v), q1 = vfma(u1, u1, v1 * v1);
        const f2 den = f2{P::fsqrt(q0.x), P::fsqrt(q0.y)} + f2{P::fsqrt(q1.x), P::fsqrt(q1.y)};
        const f2 num = vfma(du, u + u1, dv * (v + v1));
        const float da = den.x > 0.0f ? num.x * P::rcp(den.x) : 0.0f;
        s0 = da * da;
        s1 = q1.x;
        s2 = dT.x * dT.x;
        s3 = T1.x * T1.x;
        if (both) {
            rout[off + 1] = {P::add(qb.x, -div[0].y, 0), P::add(qb.y, du.y, 1),
                             P::add(qb.z, dv.y, 2), P::add(qb.w, dT.y, 3)};
            bad = bad || !(P::in_range(dr1.y, 0) && P::in_range(u1.y, 1) &&
                           P::in_range(v1.y, 2) && P::in_range(T1.y, 3));
            const float db = den.y > 0.0f ? num.y * P::rcp(den.y) : 0.0f;
            s0 = fmaf(db, db, s0);
            s1 += q1.y;
            s2 = fmaf(dT.y, dT.y, s2);
            s3 = fmaf(T1.y, T1.y, s3);
        }
    }
    const float sum = rtlbfs::warp_sum4(bad ? NAN : s0, s1, s2, s3);
    if ((tid & 7) == 0) sm.red[warp][lane >> 3] = sum;
    __syncthreads();
    rtlbfs::add_sums(sm.red, NT / 32, run->acc[slot3]);  // the next launch tests them
}

}  // namespace rtlbfsc
