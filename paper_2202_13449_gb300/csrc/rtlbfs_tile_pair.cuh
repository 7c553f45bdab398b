// rtlbfs_tile_pair.cuh -- one FP32 tile of a step in packed pairs of adjacent
// columns (the body of the FP32 tile kernels; FP64: rtlbfs_tile.cuh).
//
// A small mesh's step is one block's chain of loads, phases and barriers; a
// large one's is the instructions of all.  Against one column at a time:
//   - the arithmetic of two columns in one instruction (588 thread
//     instructions per cell-update at 512^2, overheads included, were 829);
//   - a warp evaluates one x- or y-face pair where the mesh leaves an SM one
//     tile (four times the warps a block), two or four elsewhere;
//   - ghost columns hold mirrored values two deep, so gradients need no rule
//     for them, and mirror rules are selected, not branched to;
//   - the descriptor is read from shared memory.
// 64^2 5.95 -> 3.45 us per step, 128^2 6.3 -> 3.7, 301x203 6.30 -> 5.5,
// 1024x512 19.2 -> 18.7, 512^2 10.4 -> 10.5 (bound by the launch and the
// barriers of four blocks in step); TLBFS 512^2 14.7 -> 12.7.
#pragma once

#include <cuda_runtime.h>

#include "rtlbfs_pair.cuh"

namespace rtlbfs {

// Two f2 in one 16-byte shared-memory word: (rho, u) or (v, T) of a pair.
struct alignas(16) Duo {
    f2 p, q;
};

template <int TX, int TY, int NT>
struct TileSmem<StoreQ, TX, TY, NT> {
    static constexpr int PX = TX / 2;      // pairs of a tile row
    static constexpr int NP = PX + 2;      // with the 2-cell halo
    static constexpr int BX = TX + 4, BY = TY + 4, GY = TY + 2;
    // (rho - 1, u) and (v, T - T_tile) of the haloed tile, its gradients and
    // fluxes: consecutive lanes read consecutive 16-byte words
    Duo val[2][BY][NP];
    Duo gx[2][GY][NP];
    Duo gy[2][GY][NP];
    Duo fx[2][TY][PX + 1];
    Duo fy[2][TY + 1][PX];
    // the stored records of the tile's own cells, as loaded: the update adds
    // its increments to them.  Only where they leave room for four resident
    // blocks per SM (up to 14 rows); elsewhere the update re-reads them (L2).
    static constexpr bool kRaw = TY <= 14;
    Rec raw[2][kRaw ? TY : 1][kRaw ? PX : 1];
    float xl[7][TX + 2];        // FaceLine fields of the x-faces (and one to pair the last)
    FaceLine<float> yl[TY + 1];
    float xis[BX], xdt[BX];     // CellLine is_next, dt_w of the box columns
    float yis[BY], ydt[BY];
    float red[NT / 32][4];      // per-warp residual partials (tile_sums adds them)
    CavityDesc desc;            // the tile's cavity, staged by stage_tile
    int plan[3];                // the tile's step after its cavity's stop test: done, cur, sum slot
    int last;                   // persistent kernel: this block finalises the step
};

// The mesh lines of a tile and its halo into shared memory.
template <int TX, int TY, int NT>
__device__ __forceinline__ void stage_lines(TileSmem<StoreQ, TX, TY, NT>& sm, const CavityDesc* gdp,
                                            int i0, int j0)
{
    using Sm = TileSmem<StoreQ, TX, TY, NT>;
    const int tid = threadIdx.x;
    const int nx = gdp->nx, ny = gdp->ny;
    const CellLine<float>* xc = static_cast<const CellLine<float>*>(gdp->xcell);
    const CellLine<float>* yc = static_cast<const CellLine<float>*>(gdp->ycell);
    const FaceLine<float>* xl = static_cast<const FaceLine<float>*>(gdp->xline);
    const FaceLine<float>* yl = static_cast<const FaceLine<float>*>(gdp->yline);
    for (int k = tid; k < Sm::BX; k += NT) {
        const CellLine<float> c = xc[min(i0 + k, nx + 3)];
        sm.xis[k] = c.is_next;
        sm.xdt[k] = c.dt_w;
    }
    for (int k = tid; k < Sm::BY; k += NT) {
        const CellLine<float> c = yc[min(j0 + k, ny + 3)];
        sm.yis[k] = c.is_next;
        sm.ydt[k] = c.dt_w;
    }
    for (int k = tid; k < TX + 2; k += NT) {
        const FaceLine<float> f = xl[min(i0 + k, nx)];
        sm.xl[0][k] = f.h;
        sm.xl[1][k] = f.cL;
        sm.xl[2][k] = f.cR;
        sm.xl[3][k] = f.m_nu_2h;
        sm.xl[4][k] = f.m_chi_2h;
        sm.xl[5][k] = f.m_tf15;
        sm.xl[6][k] = f.m_tg15;
    }
    for (int k = tid; k < TY + 1; k += NT) sm.yl[k] = yl[min(j0 + k, ny)];
}

// tile_step (rtlbfs_tile.cuh) for FP32.  The warps share out the faces by
// rows: a warp's 32 lanes are two rows of 16 pairs, and the remainders (the
// tile's east column and north row of faces) are one more warp's work each,
// so with TY / 2 + 1 warps every warp evaluates one packed x-face and one
// packed y-face, with twice as many one of the two, with half two of each.
template <int TX, int TY, int NT, int SCHEME, bool LDCG>
__device__ __forceinline__ void tile_step_pair(TileSmem<StoreQ, TX, TY, NT>& sm,
                                               int i0, int j0, const Rec* __restrict__ fin,
                                               Rec* __restrict__ fout)
{
    using Sm = TileSmem<StoreQ, TX, TY, NT>;
    using P = StoreQ;
    constexpr int PX = Sm::PX, NP = Sm::NP, BY = Sm::BY, GY = Sm::GY;
    constexpr int NW = NT / 32;
    static_assert(PX == 16 && TY % 2 == 0 && NT % 32 == 0, "a warp takes two rows of pairs");
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const CavityDesc& d = sm.desc;
    const int nx = d.nx, ny = d.ny, pitch = d.pitch;
    const bool xper = d.kind[kSideW] == kPeriodic, yper = d.kind[kSideS] == kPeriodic;
    const bool hlo = d.kind[kSideS] == kHalo, hhi = d.kind[kSideN] == kHalo;
    // temperature reference of this tile: its (clamped) centre cell
    const int ic = min(i0 + TX / 2, nx - 1), jc = min(j0 + TY / 2, ny - 1);
    const int qTz = ld_state<LDCG>(&fin[(size_t)jc * pitch + ic]).w;
    const float Tz = P::val(qTz, 3);
    const f2 Tz2 = splat(Tz);

    // A tile whose halo lies inside the mesh touches no boundary: no ghost
    // resolution, no mirror rules, no wall faces (block-uniform).
    const bool interior = i0 >= 2 && j0 >= 2 && i0 + TX + 2 <= nx && j0 + TY + 2 <= ny;

    // ---- 1. the haloed tile ---------------------------------------------
    {
        constexpr int NB = NP * BY, NL = (NB + NT - 1) / NT;
        Rec a[NL], b[NL];
        int ym[NL], ma[NL], mb[NL];  // mirror sides: row, column a, column b (m1 | m2 << 8)
        bool oka[NL], okb[NL];
#pragma unroll
        for (int k = 0; k < NL; ++k) {  // issue every load first
            const int t = tid + k * NT, br = t / NP, bp = t - br * NP;
            const int gi = i0 - 2 + 2 * bp, gj = j0 - 2 + br;
            if (interior) {
                if (t < NB) {
                    const Rec* p = &fin[(size_t)gj * pitch + gi];
                    if constexpr (LDCG) {
                        a[k] = ld_state<true>(p);
                        b[k] = ld_state<true>(p + 1);
                    } else {
                        ld2(p, a[k], b[k]);
                    }
                }
            } else {
                int rs, sa, sb, a2, b2;
                const bool row = t < NB && row_source(gj, ny, yper, hlo, hhi, rs, ym[k]);
                oka[k] = column_source(gi, nx, xper, sa, ma[k], a2) && row;
                okb[k] = column_source(gi + 1, nx, xper, sb, mb[k], b2) && row;
                ma[k] = (ma[k] & 0xff) | (a2 << 8);
                mb[k] = (mb[k] & 0xff) | (b2 << 8);
                a[k] = b[k] = {0, 0, 0, 0};
                const Rec* src = fin + (long long)rs * pitch;
                if (oka[k]) a[k] = ld_state<LDCG>(src + sa);
                if (okb[k]) b[k] = ld_state<LDCG>(src + sb);
            }
        }
#pragma unroll
        for (int k = 0; k < NL; ++k) {
            const int t = tid + k * NT, br = t / NP, bp = t - br * NP;
            if (t >= NB) continue;
            if constexpr (Sm::kRaw) {
                if (br >= 2 && br < TY + 2 && bp >= 1 && bp <= PX) {
                    sm.raw[0][br - 2][bp - 1] = a[k];
                    sm.raw[1][br - 2][bp - 1] = b[k];
                }
            }
            f2 v[4];
            convert2(a[k], b[k], qTz, v);
            if (!interior) {
                float wa[4] = {v[0].x, v[1].x, v[2].x, v[3].x};
                float wb[4] = {v[0].y, v[1].y, v[2].y, v[3].y};
                mirror_column(d, Tz, oka[k], ym[k], (signed char)ma[k], ma[k] >> 8, wa);
                mirror_column(d, Tz, okb[k], ym[k], (signed char)mb[k], mb[k] >> 8, wb);
#pragma unroll
                for (int q = 0; q < 4; ++q) v[q] = {wa[q], wb[q]};
            }
            sm.val[0][br][bp] = {v[0], v[1]};
            sm.val[1][br][bp] = {v[2], v[3]};
        }
    }
    __syncthreads();

    auto take = [](const Duo& a, const Duo& b, f2 v[4]) {
        v[0] = a.p;
        v[1] = a.q;
        v[2] = b.p;
        v[3] = b.q;
    };

    // ---- 2. gradients on the tile plus a 1-cell ring (Eqs. 55-56) -------
    for (int t = tid; t < NP * GY; t += NT) {
        const int gr = t / NP, gp = t - gr * NP;
        // a wall ghost row takes its partner's gradient, mirrored (ghost
        // columns need no rule: their values are mirrored two deep)
        int r = gr + 1, ym = -1;
        if (!interior && !yper) {
            if (j0 - 2 + r == -1 && !hlo) ym = kSideS;
            if (j0 - 2 + r == ny && !hhi) ym = kSideN;
            r += ym == kSideS ? 1 : (ym == kSideN ? -1 : 0);
        }
        f2 v[4], n[4], s[4], w[4], e[4], gx[4], gy[4];
        take(sm.val[0][r][gp], sm.val[1][r][gp], v);
        take(sm.val[0][r + 1][gp], sm.val[1][r + 1][gp], n);
        take(sm.val[0][r - 1][gp], sm.val[1][r - 1][gp], s);
        // neighbours of the ring's outer columns are not read by any face
        const int wp = max(gp - 1, 0), ep = min(gp + 1, NP - 1);
        take(sm.val[0][r][wp], sm.val[1][r][wp], w);
        take(sm.val[0][r][ep], sm.val[1][r][ep], e);
        const float i0w = sm.xis[max(2 * gp - 1, 0)], i1 = sm.xis[2 * gp], i2 = sm.xis[2 * gp + 1];
        const f2 in = splat(sm.yis[r]), is = splat(sm.yis[r - 1]);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const float d1 = (v[k].y - v[k].x) * i1;
            gx[k] = {fmaf(v[k].x - w[k].y, i0w, d1), fmaf(e[k].x - v[k].y, i2, d1)};
            gy[k] = vfma(n[k] - v[k], in, (v[k] - s[k]) * is);
        }
        if (ym >= 0) mirror_grad_rows(d.kind[ym], gx, gy);
        sm.gx[0][gr][gp] = {gx[0], gx[1]};
        sm.gx[1][gr][gp] = {gx[2], gx[3]};
        sm.gy[0][gr][gp] = {gy[0], gy[1]};
        sm.gy[1][gr][gp] = {gy[2], gy[3]};
    }
    __syncthreads();

    // ---- 3. faces ----------------------------------------------------
    // Tasks of a warp: x-faces west of a and between a and b, then y-faces
    // below a and b.  Task k < TY / 2 of each: rows 2k, 2k + 1; task TY / 2:
    // the remainder (the east column's faces, one row a lane; the north
    // row's).
    constexpr int TASKS = TY / 2 + 1;
    for (int task = warp; task < 2 * TASKS; task += NW) {
        const bool isx = task < TASKS;
        const int k = isx ? task : task - TASKS;
        if (isx) {
            const int row = k < TY / 2 ? 2 * k + (lane >> 4) : lane, p = k < TY / 2 ? lane & 15 : PX;
            if (row >= TY) continue;
            f2 vl[4], gxl[4], gyl[4], vr[4], gxr[4], gyr[4], F[4];
            take(sm.val[0][row + 2][p + 1], sm.val[1][row + 2][p + 1], vr);
            take(sm.gx[0][row + 1][p + 1], sm.gx[1][row + 1][p + 1], gxr);
            take(sm.gy[0][row + 1][p + 1], sm.gy[1][row + 1][p + 1], gyr);
            {  // left cells: the pair to the west's b, and a
                f2 w[4];
                take(sm.val[0][row + 2][p], sm.val[1][row + 2][p], w);
    #pragma unroll
                for (int q = 0; q < 4; ++q) vl[q] = {w[q].y, vr[q].x};
                take(sm.gx[0][row + 1][p], sm.gx[1][row + 1][p], w);
    #pragma unroll
                for (int q = 0; q < 4; ++q) gxl[q] = {w[q].y, gxr[q].x};
                take(sm.gy[0][row + 1][p], sm.gy[1][row + 1][p], w);
    #pragma unroll
                for (int q = 0; q < 4; ++q) gyl[q] = {w[q].y, gyr[q].x};
            }
            auto line = [&](int c) -> f2 { return *reinterpret_cast<const f2*>(&sm.xl[c][2 * p]); };
            FaceLine<f2> fl;
            fl.h = line(0);
            fl.cL = line(1);
            fl.cR = line(2);
            fl.m_nu_2h = line(3);
            fl.m_chi_2h = line(4);
            fl.m_tf15 = line(5);
            fl.m_tg15 = line(6);
            const int gi = i0 + 2 * p;
            faces2<true, SCHEME>(vl, gxl, gyl, vr, gxr, gyr, Tz2, fl,
                                 [&](f2& mn, f2& mt, f2 rho) {
                                     if (interior || xper) return;  // block-uniform
                                     if (gi == 0 || gi == nx) {
                                         mn.x = 0.0f;
                                         mt.x = rho.x * d.f_bcU[gi == 0 ? kSideW : kSideE];
                                     }
                                     if (gi + 1 == nx) {
                                         mn.y = 0.0f;
                                         mt.y = rho.y * d.f_bcU[kSideE];
                                     }
                                 },
                                 F);
            sm.fx[0][row][p] = {F[0], F[1]};
            sm.fx[1][row][p] = {F[2], F[3]};
        } else {
            const int row = k < TY / 2 ? 2 * k + (lane >> 4) : TY, p = k < TY / 2 ? lane & 15 : lane;
            if (p >= PX) continue;
            f2 vl[4], gxl[4], gyl[4], vr[4], gxr[4], gyr[4], F[4];
            take(sm.val[0][row + 1][p + 1], sm.val[1][row + 1][p + 1], vl);
            take(sm.gx[0][row][p + 1], sm.gx[1][row][p + 1], gxl);
            take(sm.gy[0][row][p + 1], sm.gy[1][row][p + 1], gyl);
            take(sm.val[0][row + 2][p + 1], sm.val[1][row + 2][p + 1], vr);
            take(sm.gx[0][row + 1][p + 1], sm.gx[1][row + 1][p + 1], gxr);
            take(sm.gy[0][row + 1][p + 1], sm.gy[1][row + 1][p + 1], gyr);
            const int gj = j0 + row;
            faces2<false, SCHEME>(vl, gxl, gyl, vr, gxr, gyr, Tz2, splat_line(sm.yl[row]),
                                  [&](f2& mn, f2& mt, f2 rho) {
                                      if (interior || yper) return;  // block-uniform
                                      const int ws = (gj == 0 && !hlo)    ? kSideS
                                                     : (gj == ny && !hhi) ? kSideN
                                                                          : -1;
                                      if (ws >= 0) {
                                          mn = splat(0.0f);
                                          mt = rho * splat(d.f_bcU[ws]);
                                      }
                                  },
                                  F);
            sm.fy[0][row][p] = {F[0], F[1]};
            sm.fy[1][row][p] = {F[2], F[3]};
        }
    }
    __syncthreads();

    // ---- 4. update (increment form), 5. residual sums ---------------
    PairSums acc;
    {
        const float dt = d.f_dt, sfx = d.f_fx * dt, sfy = d.f_fy * dt;
        const float sbg = d.f_beta_g * dt, Tr = d.f_T_ref;
        for (int t = tid; t < PX * TY; t += NT) {
            const int row = t / PX, p = t % PX;
            const int gi = i0 + 2 * p, gj = j0 + row;
            if (gi >= nx || gj >= ny) continue;
            f2 v[4], Fw[4], Fs[4], Fn[4], div[4];
            take(sm.val[0][row + 2][p + 1], sm.val[1][row + 2][p + 1], v);
            take(sm.fx[0][row][p], sm.fx[1][row][p], Fw);
            const Duo e0 = sm.fx[0][row][p + 1], e1 = sm.fx[1][row][p + 1];
            const float Fe[4] = {e0.p.x, e0.q.x, e1.p.x, e1.q.x};
            take(sm.fy[0][row][p], sm.fy[1][row][p], Fs);
            take(sm.fy[0][row + 1][p], sm.fy[1][row + 1][p], Fn);
            const f2 ax = {sm.xdt[2 * p + 2], sm.xdt[2 * p + 3]}, ay = splat(sm.ydt[row + 2]);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const f2 dF = {Fw[q].y - Fw[q].x, Fe[q] - Fw[q].y};
                div[q] = vfma(ax, dF, ay * (Fn[q] - Fs[q]));
            }
            const size_t o = (size_t)gj * pitch + gi;
            const bool both = gi + 1 < nx;
            Rec qa, qb;
            if constexpr (Sm::kRaw) {
                qa = sm.raw[0][row][p];
                qb = sm.raw[1][row][p];
            } else {
                qa = ld_state<LDCG>(fin + o);  // the row is padded to 32 cells: b can be read
                qb = ld_state<LDCG>(fin + o + 1);
            }
            update2(v, Tz, div, sfx, sfy, sbg, Tr, qa, qb, both, fout + o, acc);
        }
    }
    const float sum = warp_total(acc);  // FP32 within a tile, FP64 across tiles
    if ((lane & 7) == 0) sm.red[warp][lane >> 3] = sum;
}

}  // namespace rtlbfs
