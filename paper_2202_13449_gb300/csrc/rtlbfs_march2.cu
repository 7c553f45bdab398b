// rtlbfs_march2.cu -- the FP32 RTLBFS step as a warp-marching stencil, two
// adjacent columns per lane in packed FP32x2 arithmetic.
//
// Work unit: one warp, a strip of kStrip2 = 60 interior columns and a chunk
// of rows [j0, j1) of one cavity.  Lane l holds columns c0 - 2 + 2l and
// c0 - 1 + 2l: lanes 0 and 31 are the 2-cell halo, lanes 1-30 the interior.
// The warp walks up the chunk keeping a rolling window in registers --
// values of rows j and j+1, gradients of row j, the scaled difference and
// the flux through the face between rows -- and per row:
//   x-faces of row j: each lane its two cells' west faces; the left cell of
//     the first is lane l-1's second column (shuffles),
//   row j+2 (loaded one row ahead), Green-Gauss gradients of row j+1,
//   the y-faces between rows j and j+1 (all in the lane's registers),
//   the update of row j (the second cell's east face is lane l+1's first)
//     and the residual sums.
// No shared memory, no block barriers; every face is computed once (plus the
// strip-edge halo); HBM sees one read and one write of the state per cell.
//
// Why two columns a lane: the step is bound by instruction issue and the FMA
// pipe.  A packed instruction does two columns' operation in one issue slot;
// only one of a pair's two x-neighbours needs a shuffle; 4 of 64 columns are
// halo instead of 4 of 32.  Per cell 406 thread instructions instead of the
// 727 of a scalar march with one column a lane; the FMA pipe is the bound
// (a packed FMA holds it for two cycles), about 70 % busy at 4096^2: 476 ->
// 351 us per step there (35 -> 48 G cell-updates/s), 1024^2 42 -> 36 us.
// One warp a block: twelve fit an SM without spills (168 registers), where
// blocks of four warps compile to 220 registers and eight warps.
// A row's raw records come by asynchronous copies into a ring in shared
// memory: no registers hold them until the update needs them again, and the
// latency of four rows is in flight.
//
// Columns beyond a wall hold mirrored values two deep: the Green-Gauss
// gradient of the ghost column is then the mirror of its partner's, with no
// rule of its own.  Ghost rows mirror gradients explicitly.
#include <cuda_runtime.h>

#include <cmath>

#include "rtlbfs_dev.cuh"
#include "rtlbfs_kernels.h"

namespace rtlbfs {

namespace {

using P = StoreQ;
using Rec = Vec4<int>;

__device__ __forceinline__ f2 splat(float v) { return {v, v}; }

// Asynchronous global -> shared copy of a 16-byte record.
__device__ __forceinline__ void copy_async(void* dst, const void* src)
{
    const unsigned a = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(a), "l"(src) : "memory");
}
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void copy_wait()
{
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// two adjacent records at a 32-byte boundary in one access
__device__ __forceinline__ void st2(Rec* p, const Rec& a, const Rec& b)
{
    asm volatile("st.global.v8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"l"(p), "r"(a.x), "r"(a.y),
                 "r"(a.z), "r"(a.w), "r"(b.x), "r"(b.y), "r"(b.z), "r"(b.w));
}

// A column's source on a line of n cells: the cell itself, the opposite
// cell of a periodic line, or the cell that a ghost up to two beyond a wall
// mirrors (m1, then m2: the sides to mirror across, -1: none).  Columns that
// no stencil uses give false.
__device__ __forceinline__ bool column_source(int c, int n, bool per, int& src, int& m1, int& m2)
{
    m1 = m2 = -1;
    src = c;
    if (c >= 0 && c < n) return true;
    if (per) {
        src = ((c % n) + n) % n;
        return true;
    }
    if (c < -2 || c > n + 1) return false;
    if (c < 0) {
        m1 = kSideW;
        src = -1 - c;
        if (src >= n) {  // a line of one cell: the partner is itself a ghost
            m2 = m1;
            m1 = kSideE;
            src = 2 * n - 1 - src;
        }
    } else {
        m1 = kSideE;
        src = 2 * n - 1 - c;
        if (src < 0) {
            m2 = m1;
            m1 = kSideW;
            src = -1 - src;
        }
    }
    return true;
}

// Ghost values across wall `side` from the partner's working values (rho - 1,
// u, v, T - Tref): rho even, velocity odd about the wall velocity (normal
// component about 0), T odd about T_wall on a Dirichlet wall, even on an
// adiabatic one.
__device__ __forceinline__ void mirror_values2(const CavityDesc* d, int side, float Tref, float v[4])
{
    const float ut2 = 2.0f * P::bcU(d, side);
    if (side == kSideW || side == kSideE) {
        v[1] = -v[1];
        v[2] = ut2 - v[2];
    } else {
        v[2] = -v[2];
        v[1] = ut2 - v[1];
    }
    if (d->kind[side] == kDirichlet) v[3] = 2.0f * (P::Tw(d, side) - Tref) - v[3];
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
    for (int k = 0; k < 4; ++k) v[k] = x[k] * splat(P::scale_f(k));
}

// Constants of a pair of faces.
struct Line2 {
    f2 h, cL, cR, m_nu_2h, m_chi_2h, m_tf15, m_tg15;
};

// What a warp keeps in shared memory; every lane reads back only what it
// wrote or copied itself, so no synchronisation is needed.
// line: the x-face constants, the same for every row.
// row: a ring of raw rows, kAhead rows copied ahead of their use; a row stays
// until its update, which adds its increments to the stored records.
constexpr int kAhead = 4, kRing = 8;
static_assert(kRing >= kAhead + 3 && (kRing & (kRing - 1)) == 0, "rows j .. j + 2 + kAhead live");
struct WarpSmem {
    Rec row[kRing][2][32];
    f2 line[7][32];
};

// Fluxes of two faces with the same orientation from the cells on either
// side (working values v, gradients along x and y in storage order): F =
// (mass, x-, y-momentum, energy).  ISX: x-faces (normal u, tangential v).
template <bool ISX, class W>
__device__ __forceinline__ void faces2(const f2 vl[4], const f2 gxl[4], const f2 gyl[4],
                                       const f2 vr[4], const f2 gxr[4], const f2 gyr[4], f2 Tz,
                                       const Line2& ln, W wall, f2 F[4])
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
    FaceLine<f2> fl;
    fl.h = ln.h;
    fl.cL = ln.cL;
    fl.cR = ln.cR;
    fl.m_nu_2h = ln.m_nu_2h;
    fl.m_chi_2h = ln.m_chi_2h;
    fl.m_tf15 = ln.m_tf15;
    fl.m_tg15 = ln.m_tg15;
    // temperatures relative to the left cell's (its own deviation is 0)
    const f2 Tbar = Tz + L.q[3];
    f2 A[4], Na[4], M[4], D[4], B[4], Sb[4], G[4];
    R.q[3] = R.q[3] - L.q[3];
    L.q[3] = splat(0.0f);
    face_columns<f2>(L, R, fl, A, Na, M, D, B, Sb);
    face_flux_wall<f2>(A, Na, M, D, B, Sb, Tbar, fl, wall, G);
    F[0] = G[0];
    F[N] = G[1];
    F[S] = G[2];
    F[3] = G[3];
}

__device__ __forceinline__ float up1(float v) { return __shfl_up_sync(0xffffffffu, v, 1); }
__device__ __forceinline__ float dn1(float v) { return __shfl_down_sync(0xffffffffu, v, 1); }

}  // namespace

__global__ void __launch_bounds__(kMarch2Threads, kMarch2Blocks)
march2_kernel(const CavityDesc* __restrict__ descs, CavityRun* __restrict__ runs,
              const int4* __restrict__ units, const int* __restrict__ nunits_ptr, int par)
{
    const int lane = threadIdx.x & 31;
    constexpr int wpb = kMarch2Threads / 32;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    WarpSmem& sm = reinterpret_cast<WarpSmem*>(smem_raw)[threadIdx.x >> 5];
    chain_sync();
    const int nunits = *nunits_ptr;

    for (int ui = blockIdx.x * wpb + (threadIdx.x >> 5); ui < nunits; ui += gridDim.x * wpb) {
        const int4 wu = units[ui];
        const int slot = wu.x, c0 = wu.y, j0 = wu.z, j1 = wu.w;
        const CavityDesc* dp = descs + slot;
        CavityRun* run = runs + slot;
        // the stop test of the cavity's previous step (lane 0; the cavity's
        // first unit also publishes the header for the next launch)
        int plan = 0;
        if (lane == 0) {
            const CavityCtl d = run_head(run, par);
            if (ui == dp->tile_begin) run_publish(run, par, d);
            plan = d.done | (d.cur << 1) | ((int)(d.steps % 3) << 2);
        }
        plan = __shfl_sync(0xffffffffu, plan, 0);
        if (plan & 1) continue;  // warp-uniform
        const int cur = (plan >> 1) & 1, slot3 = plan >> 2;
        const int nx = dp->nx, ny = dp->ny, pitch = dp->pitch;
        const bool xper = dp->kind[kSideW] == kPeriodic, yper = dp->kind[kSideS] == kPeriodic;
        const bool hlo = dp->kind[kSideS] == kHalo, hhi = dp->kind[kSideN] == kHalo;
        // south / north sides that are walls (not periodic, not a strip's halo)
        const bool wall_s = !yper && !hlo, wall_n = !yper && !hhi;
        const Rec* __restrict__ fin = static_cast<const Rec*>(dp->f[cur][0]);
        Rec* __restrict__ fout = static_cast<Rec*>(dp->f[cur ^ 1][0]);
        const CellLine<float>* xc = static_cast<const CellLine<float>*>(dp->xcell);
        const CellLine<float>* yc = static_cast<const CellLine<float>*>(dp->ycell);
        const FaceLine<float>* xl = static_cast<const FaceLine<float>*>(dp->xline);
        const FaceLine<float>* yl = static_cast<const FaceLine<float>*>(dp->yline);

        // this lane's two columns a = ga, b = ga + 1
        const int ga = c0 - 2 + 2 * lane;
        // every column of the strip and its halo inside the mesh (warp-uniform)
        const bool inside = c0 >= 2 && c0 + kStrip2 + 2 <= nx;
        const bool xwall = !xper && (c0 == 0 || c0 + kStrip2 + 1 >= nx);  // may touch a wall face
        auto cell = [&](int c) { return xc[min(max(c + 2, 0), nx + 3)]; };
        const float i0 = cell(ga - 1).is_next, i1 = cell(ga).is_next;
        const f2 dtx = {cell(ga).dt_w, cell(ga + 1).dt_w};
        {
            const FaceLine<float> p = xl[min(max(ga, 0), nx)], q = xl[min(max(ga + 1, 0), nx)];
            sm.line[0][lane] = {p.h, q.h};
            sm.line[1][lane] = {p.cL, q.cL};
            sm.line[2][lane] = {p.cR, q.cR};
            sm.line[3][lane] = {p.m_nu_2h, q.m_nu_2h};
            sm.line[4][lane] = {p.m_chi_2h, q.m_chi_2h};
            sm.line[5][lane] = {p.m_tf15, q.m_tf15};
            sm.line[6][lane] = {p.m_tg15, q.m_tg15};
        }
        const bool upd_a = lane >= 1 && lane <= 30 && ga < nx, upd_b = upd_a && ga + 1 < nx;

        // Eq. 64's source over the density, times the time step
        const float dtc = P::dt(dp), sfx = P::fx(dp) * dtc, sfy = P::fy(dp) * dtc;
        const float sbg = P::beta_g(dp) * dtc, Tr = P::T_ref(dp);
        // temperature reference of this unit
        const int qTz = fin[(size_t)min(j0, ny - 1) * pitch + min(c0 + 30, nx - 1)].w;
        const float Tz = P::val(qTz, 3);
        const f2 Tz2 = splat(Tz);

        // raw records of row r (a ghost row: its partner's), ghost rules
        // applied later in values()
        auto row_source = [&](int r, int& rs, int& ym) -> bool {
            ym = -1;
            rs = r;
            if ((r >= 0 && r < ny) || (r < 0 && hlo && r >= -2) || (r >= ny && hhi && r <= ny + 1))
                return true;
            if (yper) {
                rs = ((r % ny) + ny) % ny;
                return true;
            }
            if (r == -1) {
                rs = 0;
                ym = kSideS;
                return true;
            }
            if (r == ny) {
                rs = ny - 1;
                ym = kSideN;
                return true;
            }
            return false;
        };
        // the records this lane's columns take their values from (a column
        // that no stencil uses: any record)
        int sa, sb;
        {
            int m1, m2;
            if (!column_source(ga, nx, xper, sa, m1, m2)) sa = 0;
            if (!column_source(ga + 1, nx, xper, sb, m1, m2)) sb = 0;
        }
        auto fetch = [&](int r) {
            int rs, ym;
            if (r <= j1 + 1) {
                if (!row_source(r, rs, ym)) rs = 0;
                const Rec* row = fin + (long long)rs * pitch;
                copy_async(&sm.row[r & (kRing - 1)][0][lane], row + sa);
                copy_async(&sm.row[r & (kRing - 1)][1][lane], row + sb);
            }
        };
        auto values = [&](int r, f2 v[4]) {
            convert2(sm.row[r & (kRing - 1)][0][lane], sm.row[r & (kRing - 1)][1][lane], qTz, v);
            int rs, ym;
            const bool ok = row_source(r, rs, ym);
            if (inside && ym < 0 && ok) return;  // warp-uniform
            auto ghost = [&](int c, float w[4]) {
                int s, m1, m2;
                if (!ok || !column_source(c, nx, xper, s, m1, m2)) {
                    w[0] = w[1] = w[2] = w[3] = 0.0f;
                    return;
                }
                if (ym >= 0) mirror_values2(dp, ym, Tz, w);
                if (m1 >= 0) mirror_values2(dp, m1, Tz, w);
                if (m2 >= 0) mirror_values2(dp, m2, Tz, w);
            };
            float wa[4] = {v[0].x, v[1].x, v[2].x, v[3].x}, wb[4] = {v[0].y, v[1].y, v[2].y, v[3].y};
            ghost(ga, wa);
            ghost(ga + 1, wb);
#pragma unroll
            for (int k = 0; k < 4; ++k) v[k] = {wa[k], wb[k]};
        };
        // Green-Gauss d/dx of a row (Eqs. 55-56) from neighbour differences
        auto grad_x = [&](const f2 v[4], f2 g[4]) {
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const float s0 = (v[k].x - up1(v[k].y)) * i0, s1 = (v[k].y - v[k].x) * i1;
                const float s2 = dn1(s0);
                g[k] = {s0 + s1, s1 + s2};
            }
        };
        // 1 / (w + w_next) between rows r and r + 1
        auto is_row = [&](int r) { return splat(yc[min(max(r + 2, 0), ny + 3)].is_next); };
        // y-faces between rows jf - 1 (l) and jf (r)
        auto yfaces = [&](int jf, const FaceLine<float>& p, const f2 vl[4], const f2 gxl[4], const f2 gyl[4], const f2 vr[4],
                          const f2 gxr[4], const f2 gyr[4], f2 F[4]) {
            const Line2 ly = {splat(p.h), splat(p.cL), splat(p.cR), splat(p.m_nu_2h),
                              splat(p.m_chi_2h), splat(p.m_tf15), splat(p.m_tg15)};
            const int ws = (wall_s && jf == 0) ? kSideS : ((wall_n && jf == ny) ? kSideN : -1);
            faces2<false>(vl, gxl, gyl, vr, gxr, gyr, Tz2, ly,
                          [&](f2& mn, f2& mt, f2 rho) {
                              if (ws >= 0) {  // warp-uniform
                                  mn = splat(0.0f);
                                  mt = rho * splat(P::bcU(dp, ws));
                              }
                          },
                          F);
        };

        // ---- prologue: rows j0-2 .. j0+1, gradients of j0-1 and j0, the
        //      faces below row j0, copies of the rows after
        f2 v0[4], v1[4], gx0[4], gy0[4], tc[4], Fs[4];
        {
            for (int r = j0 - 2; r < j0 + 2; ++r) fetch(r);
            copy_commit();
            for (int r = j0 + 2; r < j0 + 2 + kAhead; ++r) {
                fetch(r);
                copy_commit();
            }
            f2 vm2[4], vm[4], gxm[4], gym[4];
            copy_wait<kAhead>();
            values(j0 - 2, vm2);
            values(j0 - 1, vm);
            values(j0, v0);
            values(j0 + 1, v1);
            grad_x(vm, gxm);
            grad_x(v0, gx0);
            const f2 i2 = is_row(j0 - 2), i3 = is_row(j0 - 1), i4 = is_row(j0);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const f2 a = (vm[k] - vm2[k]) * i2, b = (v0[k] - vm[k]) * i3;
                tc[k] = (v1[k] - v0[k]) * i4;
                gym[k] = a + b;
                gy0[k] = b + tc[k];
            }
            if (wall_s && j0 == 0) {  // row -1 is the south ghost: mirror row 0
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    gxm[k] = gx0[k];
                    gym[k] = gy0[k];
                }
                mirror_grad_rows(dp->kind[kSideS], gxm, gym);
            }
            yfaces(j0, yl[min(max(j0, 0), ny)], vm, gxm, gym, v0, gx0, gy0, Fs);
        }

        f2 s0 = splat(0.0f), s1 = s0, s2 = s0, s3 = s0;
        bool bad = false;

        for (int j = j0; j < j1; ++j) {
            // this row's line constants, asked for before they are needed
            const FaceLine<float> fly = yl[min(j + 1, ny)];
            const f2 in = is_row(j + 1);
            const float dty = yc[j + 2].dt_w;
            // x-faces of row j: left cells (lane l-1's b, a), right cells (a, b)
            f2 dF[4];
            {
                f2 vl[4], gxl[4], gyl[4], Fx[4];
                const Line2 lx = {sm.line[0][lane], sm.line[1][lane], sm.line[2][lane], sm.line[3][lane],
                                  sm.line[4][lane], sm.line[5][lane], sm.line[6][lane]};
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    vl[k] = {up1(v0[k].y), v0[k].x};
                    gxl[k] = {up1(gx0[k].y), gx0[k].x};
                    gyl[k] = {up1(gy0[k].y), gy0[k].x};
                }
                faces2<true>(vl, gxl, gyl, v0, gx0, gy0, Tz2, lx,
                             [&](f2& mn, f2& mt, f2 rho) {
                                 if (xwall) {  // warp-uniform
                                     const bool wa = ga == 0 || ga == nx, wb = ga + 1 == nx;
                                     if (wa) {
                                         mn.x = 0.0f;
                                         mt.x = rho.x * P::bcU(dp, ga == 0 ? kSideW : kSideE);
                                     }
                                     if (wb) {
                                         mn.y = 0.0f;
                                         mt.y = rho.y * P::bcU(dp, kSideE);
                                     }
                                 }
                             },
                             Fx);
#pragma unroll
                for (int k = 0; k < 4; ++k) dF[k] = {Fx[k].y - Fx[k].x, dn1(Fx[k].x) - Fx[k].y};
            }
            // row j+2, gradients of row j+1 (a north ghost row mirrors row j)
            f2 v2[4], gx1[4], gy1[4];
            copy_wait<kAhead - 1>();
            values(j + 2, v2);
            fetch(j + 2 + kAhead);
            copy_commit();
            grad_x(v1, gx1);
            {
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const f2 tn = (v2[k] - v1[k]) * in;
                    gy1[k] = tc[k] + tn;
                    tc[k] = tn;
                }
            }
            if (wall_n && j + 1 == ny) {
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    gx1[k] = gx0[k];
                    gy1[k] = gy0[k];
                }
                mirror_grad_rows(dp->kind[kSideN], gx1, gy1);
            }
            f2 Fn[4];
            yfaces(j + 1, fly, v0, gx0, gy0, v1, gx1, gy1, Fn);
            // update row j
            if (upd_a) {
                f2 div[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) div[k] = vfma(dtx, dF[k], splat(dty) * (Fn[k] - Fs[k]));
                const f2 dr = v0[0], u = v0[1], v = v0[2], T = Tz2 + v0[3];
                const f2 rho = splat(1.0f) + dr;
                const f2 src_x = rho * splat(sfx);
                const f2 src_y = rho * vfma(splat(sbg), T - splat(Tr), splat(sfy));
                const f2 inv = vtraits<f2>::rcp(rho - div[0]);
                const f2 du = (vfma(u, div[0], src_x) - div[1]) * inv;
                const f2 dv = (vfma(v, div[0], src_y) - div[2]) * inv;
                const f2 dT = (T * div[0] - div[3]) * inv;
                const f2 dr1 = dr - div[0], u1 = u + du, v1n = v + dv, T1 = T + dT;
                Rec* const outp = fout + (size_t)j * pitch + ga;
                const Rec qa = sm.row[j & (kRing - 1)][0][lane], qb = sm.row[j & (kRing - 1)][1][lane];
                const Rec oa = {P::add(qa.x, -div[0].x, 0), P::add(qa.y, du.x, 1),
                                P::add(qa.z, dv.x, 2), P::add(qa.w, dT.x, 3)};
                const Rec ob = {P::add(qb.x, -div[0].y, 0), P::add(qb.y, du.y, 1),
                                P::add(qb.z, dv.y, 2), P::add(qb.w, dT.y, 3)};
                const bool ba = !(P::in_range(dr1.x, 0) && P::in_range(u1.x, 1) &&
                                  P::in_range(v1n.x, 2) && P::in_range(T1.x, 3));
                const bool bb = !(P::in_range(dr1.y, 0) && P::in_range(u1.y, 1) &&
                                  P::in_range(v1n.y, 2) && P::in_range(T1.y, 3));
                const f2 q0 = vfma(u, u, v * v), q1 = vfma(u1, u1, v1n * v1n);
                const f2 den = f2{P::fsqrt(q0.x), P::fsqrt(q0.y)} + f2{P::fsqrt(q1.x), P::fsqrt(q1.y)};
                const f2 num = vfma(du, u + u1, dv * (v + v1n));
                f2 dm = {den.x > 0.0f ? num.x * P::rcp(den.x) : 0.0f,
                         den.y > 0.0f ? num.y * P::rcp(den.y) : 0.0f};
                f2 e1 = q1, e2 = dT, e3 = T1;
                bad = bad || ba || (bb && upd_b);
                if (upd_b) {
                    st2(outp, oa, ob);
                } else {  // the last column of an odd line: cell b is not a cell
                    *outp = oa;
                    dm.y = e1.y = e2.y = e3.y = 0.0f;
                }
                s0 = vfma(dm, dm, s0);
                s1 = s1 + e1;
                s2 = vfma(e2, e2, s2);
                s3 = vfma(e3, e3, s3);
            }
            // roll the window
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                Fs[k] = Fn[k];
                v0[k] = v1[k];
                v1[k] = v2[k];
                gx0[k] = gx1[k];
                gy0[k] = gy1[k];
            }
        }
        float a0 = bad ? NAN : s0.x + s0.y, a1 = s1.x + s1.y, a2 = s2.x + s2.y, a3 = s3.x + s3.y;
        const float sum = warp_sum4(a0, a1, a2, a3);
        // the step's residual sums; the next launch tests them
        if ((lane & 7) == 0) atomicAdd(&run->acc[slot3][lane >> 3], (double)sum);
        __syncwarp();
    }
}

static constexpr size_t kSmem2 = sizeof(WarpSmem) * (kMarch2Threads / 32);

// An SM's shared memory, what the system takes of it per block, and the most
// a block may ask for.
static constexpr size_t kSmemSM = 228 * 1024, kSmemSystem = 1024, kSmemMax = 227 * 1024;

cudaError_t march2_prepare()
{
    return cudaFuncSetAttribute(march2_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)kSmemMax);
}

cudaError_t march2_occupancy(int* blocks_per_sm)
{
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, march2_kernel,
                                                         kMarch2Threads, kSmem2);
}

cudaError_t launch_march2(int grid, int cap, cudaStream_t s, const CavityDesc* descs,
                          CavityRun* runs, const int4* units, const int* nunits, int par)
{
    // residency is limited by asking for just over a (cap + 1)-th of the
    // shared memory: what is left serves as L1 cache
    size_t smem = kSmem2;
    if (cap > 0) {
        const size_t share = (kSmemSM / ((size_t)cap + 1) - kSmemSystem) / 128 * 128 + 256;
        smem = share < kSmem2 ? kSmem2 : (share > kSmemMax ? kSmemMax : share);
    }
    return launch_chained(march2_kernel, grid, kMarch2Threads, smem, s, descs, runs, units, nunits,
                          par);
}

}  // namespace rtlbfs
