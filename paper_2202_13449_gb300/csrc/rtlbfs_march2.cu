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
// No block barriers; shared memory holds only what a lane reads back itself (a
// ring of raw rows, the x-face constants); every face is computed once (plus
// the strip-edge halo); HBM sees one read and one write of the state per cell.
//
// Why two columns a lane: the step is bound by instruction issue and the FMA
// pipe.  A packed instruction does two columns' operation in one issue slot;
// only one of a pair's two x-neighbours needs a shuffle; 4 of 64 columns are
// halo instead of 4 of 32.  Per cell 444 thread instructions instead of the
// 727 of a scalar march with one column a lane; the FMA pipe leads (a packed
// FMA holds it for two cycles), 61 % busy at 4096^2: 476 -> 336 us per step
// there (35 -> 50 G cell-updates/s), 1024^2 42 -> 33.5 us.
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
#include "rtlbfs_pair.cuh"
#include "rtlbfs_smem.h"

namespace rtlbfs {

namespace {

using P = StoreQ;

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

        auto row = [&](int r, int& rs, int& ym) {
            return row_source(r, ny, yper, hlo, hhi, rs, ym);
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
                if (!row(r, rs, ym)) rs = 0;
                const Rec* src = fin + (long long)rs * pitch;
                copy_async(&sm.row[r & (kRing - 1)][0][lane], src + sa);
                copy_async(&sm.row[r & (kRing - 1)][1][lane], src + sb);
            }
        };
        auto values = [&](int r, f2 v[4]) {
            convert2(sm.row[r & (kRing - 1)][0][lane], sm.row[r & (kRing - 1)][1][lane], qTz, v);
            int rs, ym;
            const bool ok = row(r, rs, ym);
            if (inside && ym < 0 && ok) return;  // warp-uniform
            auto ghost = [&](int c, float w[4]) {
                int s, m1, m2;
                const bool used = column_source(c, nx, xper, s, m1, m2) && ok;
                mirror_column(*dp, Tz, used, ym, m1, m2, w);
            };
            // (the descriptor's wall values by address: once per ghost row or edge strip)
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
            const int ws = (wall_s && jf == 0) ? kSideS : ((wall_n && jf == ny) ? kSideN : -1);
            faces2<false, 0>(vl, gxl, gyl, vr, gxr, gyr, Tz2, splat_line(p),
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

        PairSums acc;

        for (int j = j0; j < j1; ++j) {
            // this row's line constants, asked for before they are needed
            const FaceLine<float> fly = yl[min(j + 1, ny)];
            const f2 in = is_row(j + 1);
            const float dty = yc[j + 2].dt_w;
            // x-faces of row j: left cells (lane l-1's b, a), right cells (a, b)
            f2 dF[4];
            {
                f2 vl[4], gxl[4], gyl[4], Fx[4];
                const FaceLine<f2> lx = {sm.line[0][lane], sm.line[1][lane], sm.line[2][lane],
                                         sm.line[3][lane], sm.line[4][lane], sm.line[5][lane],
                                         sm.line[6][lane], splat(0.0f)};
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    vl[k] = {up1(v0[k].y), v0[k].x};
                    gxl[k] = {up1(gx0[k].y), gx0[k].x};
                    gyl[k] = {up1(gy0[k].y), gy0[k].x};
                }
                faces2<true, 0>(vl, gxl, gyl, v0, gx0, gy0, Tz2, lx,
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
                update2(v0, Tz, div, sfx, sfy, sbg, Tr, sm.row[j & (kRing - 1)][0][lane],
                        sm.row[j & (kRing - 1)][1][lane], upd_b, fout + (size_t)j * pitch + ga, acc);
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
        const float sum = warp_total(acc);
        // the step's residual sums; the next launch tests them
        if ((lane & 7) == 0) atomicAdd(&run->acc[slot3][lane >> 3], (double)sum);
        __syncwarp();
    }
}

static constexpr size_t kSmem2 = sizeof(WarpSmem) * (kMarch2Threads / 32);

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
