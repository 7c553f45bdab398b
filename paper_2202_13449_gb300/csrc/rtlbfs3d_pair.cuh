// rtlbfs3d_pair.cuh -- the FP32 3D step in packed pairs of cells adjacent
// along x (included by rtlbfs3d.cu; FP64: step3_kernel there).
//
// The same work split as step3_kernel -- a TX x TY tile of columns marches up
// a chunk of z-planes, planes k .. k+2 of values and k, k+1 of gradients in
// shared memory -- with one thread per pair of columns, whose face, gradient
// and update arithmetic runs two cells an instruction.  80^3 in 16 x 8 tiles:
// 48 us a step; a thread per cell in scalar arithmetic took 67, issue-bound at
// 3250 instructions a cell.  What bounds it now is latency: 1500 instructions
// a cell keep the schedulers busy 40 % of the time with the 8 warps that 234
// registers a thread leave room for (large meshes in 32 x 8: half of it with 12).
//  - Face fluxes change hands as registers (x: shuffles) or through shared
//    memory (y, and the tile's east column), so that three 32 x 8 blocks fit.
//  - Raw records of the plane to come are fetched after the faces, which need
//    the registers; the update covers their latency (fetched before the
//    gradients: 32 x 8 at 168 registers spilled, 165 us at 128^3 instead of 150).
//  - The planes below a chunk go through the same loop body: copies of it for
//    a prologue cost more in instruction fetches than they saved (16^3: 12.3
//    us instead of 11.6).
//
// Ghost columns along x hold values mirrored two deep, so the Green-Gauss
// gradient of a ghost column is its partner's mirror without a rule of its
// own; ghost rows and planes mirror gradients explicitly.
#pragma once

namespace rtlbfs3 {

using rtlbfs::f2;
using rtlbfs::splat;

template <int TX, int TY>
struct Smem3P {
    static constexpr int PX = TX / 2, NP = PX + 2, BY = TY + 4, GY = TY + 2, NT = PX * TY;
    f2 v[3][5][BY][NP];    // (rho - 1, u, v, w, T - Tz) of planes, 2-cell ring
    f2 g[2][15][GY][NP];   // gradients [q*3 + dir] of planes, 1-cell ring
    union {
        f2 fy[5][TY + 1][PX];   // y-face fluxes of the current plane (global components)
        double red[NT / 32][4];  // after the last plane
    };
    float zline[12];       // of the current plane: FaceLine above it, is_next, is_next above, dt_w
    f2 xl[7][PX + 1];      // FaceLine fields of the faces 2p, 2p + 1
    FaceLine<float> yl[TY + 1];
    float xisn[TX + 4], xdtw[TX + 4];  // CellLine is_next, dt_w of the ringed tile
    float yisn[BY], ydtw[BY];
    // ghost rule of side s (6: none): velocity off - vel or vel, T likewise
    float4 off[7];         // 2 u_wall (x, y, z), 2 (T_wall - Tz)
    float2 sgn[7];         // +-1: of the velocities, of T
    int plan[3];           // after the stop test: done, cur, sum slot
};

// Values and gradients of a pair of cells in the frame of axis AX.
template <int AX, int TX, int TY>
__device__ __forceinline__ void take_pair(const Smem3P<TX, TY>& sm, int vs, int gs, int r, int p,
                                          CellNT3<f2>& o)
{
    constexpr int a1 = (AX + 1) % 3, a2 = (AX + 2) % 3;
    constexpr int comp[5] = {0, 1 + AX, 1 + a1, 1 + a2, 4};
#pragma unroll
    for (int q = 0; q < 5; ++q) {
        o.q[q] = sm.v[vs][comp[q]][r][p];
        o.gn[q] = sm.g[gs][comp[q] * 3 + AX][r - 1][p];
        o.g1[q] = sm.g[gs][comp[q] * 3 + a1][r - 1][p];
        o.g2[q] = sm.g[gs][comp[q] * 3 + a2][r - 1][p];
    }
}

// Fluxes of two faces normal to axis AX between cells L and R, in global
// components (rho, x, y, z, T).
template <int AX, int SCH, class W>
__device__ __forceinline__ void face_pair(CellNT3<f2>& L, CellNT3<f2>& R, f2 Tz,
                                          const FaceLine<f2>& fl, W wall, f2 out[5])
{
    constexpr int a1 = (AX + 1) % 3, a2 = (AX + 2) % 3;
    const f2 Tbar = Tz + L.q[4];
    R.q[4] = R.q[4] - L.q[4];
    L.q[4] = splat(0.0f);
    f2 F[5];
    if constexpr (SCH == 1) {
        face_flux3_tlbfs_wall<f2>(L, R, Tbar, fl, wall, F);
    } else {
        Cols3<f2> c;
        face3_columns<f2>(L, R, fl, c);
        face_flux3_wall<f2>(c, Tbar, fl, wall, F);
    }
    out[0] = F[0];
    out[1 + AX] = F[1];
    out[1 + a1] = F[2];
    out[1 + a2] = F[3];
    out[4] = F[4];
}

// Resident blocks per SM to compile for: what the tile buffers allow, with
// 240 registers a thread in the two-warp tiles and 168 in the four-warp one.
// 168 spills about 100 bytes, which slows a lone block by a tenth, and pays
// where the mesh fills the third block: 32 x 8 at 128^3 takes 150 us with
// 12 warps per SM and 172 with 8, at 80^3 49.6 with 8 and 54 with 12; 16 x 8
// at 80^3 takes 48 us with 8 and 58 with 10.
template <int TX, int TY>
struct PairBlocks {
    static constexpr int smem = 228 * 1024 / ((int)sizeof(Smem3P<TX, TY>) + 1024);
    static constexpr int regs = 65536 / (Smem3P<TX, TY>::NT * (Smem3P<TX, TY>::NT > 64 ? 168 : 240));
    static constexpr int value = smem < regs ? smem : regs;
};

template <int TX, int TY, int SCH>
__global__ void __launch_bounds__(Smem3P<TX, TY>::NT, PairBlocks<TX, TY>::value)
step3_pair_kernel(const Desc3* __restrict__ dp, CavityRun* __restrict__ run, int par)
{
    using P = StoreQ;
    using Sm = Smem3P<TX, TY>;
    using Rec = Vec4<int>;
    constexpr int PX = Sm::PX, NP = Sm::NP, BY = Sm::BY, GY = Sm::GY, NT = Sm::NT;
    extern __shared__ __align__(16) unsigned char smraw[];
    Sm& sm = *reinterpret_cast<Sm*>(smraw);

    const int tid = threadIdx.x, px = tid % PX, ty = tid / PX, lane = tid & 31, warp = tid >> 5;
    const Desc3& d = *dp;
    const int nx = d.n[0], ny = d.n[1], nz = d.n[2];
    int u = blockIdx.x;
    const int tix = u % d.tiles_x;
    u /= d.tiles_x;
    const int tiy = u % d.tiles_y;
    const int ch = u / d.tiles_y;
    const int i0 = tix * TX, j0 = tiy * TY, k0 = ch * d.kchunk, k1 = min(nz, k0 + d.kchunk);
    const bool xper = d.kind[0] == kPeriodic, yper = d.kind[2] == kPeriodic;
    const bool zper = d.kind[4] == kPeriodic;
    const FaceLine<float>* zl = static_cast<const FaceLine<float>*>(d.fline[2]);
    const CellLine<float>* zc = static_cast<const CellLine<float>*>(d.cline[2]);
    // mesh lines: written by the host, not by the previous step, so fetched
    // before the wait
    {
        const FaceLine<float>* xl = static_cast<const FaceLine<float>*>(d.fline[0]);
        const FaceLine<float>* yl = static_cast<const FaceLine<float>*>(d.fline[1]);
        const CellLine<float>* xc = static_cast<const CellLine<float>*>(d.cline[0]);
        const CellLine<float>* yc = static_cast<const CellLine<float>*>(d.cline[1]);
        for (int t = tid; t < PX + 1; t += NT) {
            const FaceLine<float> a = xl[min(i0 + 2 * t, nx)], b = xl[min(i0 + 2 * t + 1, nx)];
            sm.xl[0][t] = {a.h, b.h};
            sm.xl[1][t] = {a.cL, b.cL};
            sm.xl[2][t] = {a.cR, b.cR};
            sm.xl[3][t] = {a.m_nu_2h, b.m_nu_2h};
            sm.xl[4][t] = {a.m_chi_2h, b.m_chi_2h};
            sm.xl[5][t] = {a.m_tf15, b.m_tf15};
            sm.xl[6][t] = {a.m_tg15, b.m_tg15};
        }
        for (int t = tid; t < TY + 1; t += NT) sm.yl[t] = yl[min(j0 + t, ny)];
        for (int t = tid; t < TX + 4; t += NT) {
            const CellLine<float> c = xc[min(i0 + t, nx + 3)];
            sm.xisn[t] = c.is_next;
            sm.xdtw[t] = c.dt_w;
        }
        for (int t = tid; t < BY; t += NT) {
            const CellLine<float> c = yc[min(j0 + t, ny + 3)];
            sm.yisn[t] = c.is_next;
            sm.ydtw[t] = c.dt_w;
        }
    }
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
    if (sm.plan[0]) return;  // uniform
    const int cur = sm.plan[1], slot3 = sm.plan[2];
    const Rec* __restrict__ rin = static_cast<const Rec*>(d.rec[cur]);
    const int* __restrict__ tin = static_cast<const int*>(d.tem[cur]);
    Rec* __restrict__ rout = static_cast<Rec*>(d.rec[cur ^ 1]);
    int* __restrict__ tout = static_cast<int*>(d.tem[cur ^ 1]);
    const long long plane = (long long)nx * ny;
    // temperature reference of this unit: one stored cell value
    const int qTz = tin[((size_t)k0 * ny + min(j0 + TY / 2, ny - 1)) * nx + min(i0 + TX / 2, nx - 1)];
    const float Tz = P::val(qTz, 3);
    const f2 Tz2 = splat(Tz);
    if (tid < 7) {
        float4 o = {0.0f, 0.0f, 0.0f, 0.0f};
        float2 s = {1.0f, 1.0f};
        if (tid < 6) {
            o = {2.0f * d.f_bcU[tid][0], 2.0f * d.f_bcU[tid][1], 2.0f * d.f_bcU[tid][2], 0.0f};
            s.x = -1.0f;
            if (d.kind[tid] == kDirichlet) {
                o.w = 2.0f * (d.f_bcT[tid] - Tz);
                s.y = -1.0f;
            }
        }
        sm.off[tid] = o;
        sm.sgn[tid] = s;
    }

    // Box items of this thread, the same for every plane: the in-plane
    // offsets of the pair's two sources, and packed sides (6: none) of the
    // row's and the columns' ghost rules with validity bits.
    constexpr int NL = (NP * BY + NT - 1) / NT;
    int oa[NL], ob[NL], rule[NL];
    bool inside = true;  // no ghost along x or y in this thread's items
#pragma unroll
    for (int k = 0; k < NL; ++k) {
        const int t = tid + k * NT, r = t / NP, p = t - r * NP;
        int js = 0, ym = -1, sa = 0, sb = 0, ma, mb, a2, b2;
        bool row = t < NP * BY;
        {
            const int j = j0 - 2 + r;
            js = j;
            if (j < 0 || j >= ny) {
                if (yper) js = ((j % ny) + ny) % ny;
                else if (j == -1 || j == ny) {
                    ym = j < 0 ? 2 : 3;
                    js = j < 0 ? 0 : ny - 1;
                } else row = false;
            }
        }
        const bool va = rtlbfs::column_source(i0 - 2 + 2 * p, nx, xper, sa, ma, a2) && row;
        const bool vb = rtlbfs::column_source(i0 - 1 + 2 * p, nx, xper, sb, mb, b2) && row;
        oa[k] = va ? js * nx + sa : 0;
        ob[k] = vb ? js * nx + sb : 0;
        auto side = [](int s) { return s < 0 ? 6 : s; };
        rule[k] = side(ym) | side(ma) << 3 | side(a2) << 6 | side(mb) << 9 | side(b2) << 12 |
                  (va ? 1 << 15 : 0) | (vb ? 1 << 16 : 0);
        inside = inside && va && vb && ym < 0 && ma < 0 && mb < 0;
        if (t >= NP * BY) rule[k] = -1;
    }
    // the raw records of the plane to store next
    Rec ra[NL], rb[NL];
    int ta[NL], tb[NL];
    auto fetch = [&](int kk) {
        int ks, zs;
        if (!resolve_1d(kk, nz, zper, 4, 5, ks, zs)) ks = 0;
        const long long base = ks * plane;
#pragma unroll
        for (int k = 0; k < NL; ++k) {
            if (rule[k] == -1) continue;
            ra[k] = rin[base + oa[k]];
            rb[k] = rin[base + ob[k]];
            ta[k] = tin[base + oa[k]];
            tb[k] = tin[base + ob[k]];
        }
    };
    // plane kk into value slot mod3(kk), ghost rules applied: z, then y, then x
    auto store = [&](int kk) {
        const int vs = mod3(kk);
        int ks, zs;
        const bool zok = resolve_1d(kk, nz, zper, 4, 5, ks, zs);
#pragma unroll
        for (int k = 0; k < NL; ++k) {
            const int t = tid + k * NT, r = t / NP, p = t - r * NP;
            if (rule[k] == -1) continue;
            const Rec a = ra[k], b = rb[k];
            const float sd = P::scale_f(0), su = P::scale_f(1), sT = P::scale_f(3);
            f2 v[5] = {f2{(float)a.x, (float)b.x} * splat(sd), f2{(float)a.y, (float)b.y} * splat(su),
                       f2{(float)a.z, (float)b.z} * splat(su), f2{(float)a.w, (float)b.w} * splat(su),
                       f2{(float)(int)((unsigned)ta[k] - (unsigned)qTz),
                          (float)(int)((unsigned)tb[k] - (unsigned)qTz)} * splat(sT)};
            if (!inside || zs >= 0 || !zok) {
                float w[2][5];
#pragma unroll
                for (int q = 0; q < 5; ++q) {
                    w[0][q] = v[q].x;
                    w[1][q] = v[q].y;
                }
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    const int s[4] = {zs < 0 ? 6 : zs, rule[k] & 7, (rule[k] >> (3 + 6 * c)) & 7,
                                      (rule[k] >> (6 + 6 * c)) & 7};
#pragma unroll
                    for (int m = 0; m < 4; ++m) {
                        if (m == 3 && s[m] == 6) continue;  // only on a line of one cell
                        const float4 o = sm.off[s[m]];
                        const float2 g = sm.sgn[s[m]];
                        w[c][1] = fmaf(g.x, w[c][1], o.x);
                        w[c][2] = fmaf(g.x, w[c][2], o.y);
                        w[c][3] = fmaf(g.x, w[c][3], o.z);
                        w[c][4] = fmaf(g.y, w[c][4], o.w);
                    }
                    const bool ok = zok && (rule[k] >> (15 + c) & 1);
#pragma unroll
                    for (int q = 0; q < 5; ++q) w[c][q] = ok ? w[c][q] : 0.0f;
                }
#pragma unroll
                for (int q = 0; q < 5; ++q) v[q] = {w[0][q], w[1][q]};
            }
#pragma unroll
            for (int q = 0; q < 5; ++q) sm.v[vs][q][r][p] = v[q];
        }
    };

    // gradients of plane kk into gradient slot mod2(kk), 1-cell ring; a
    // z-wall ghost plane mirrors the other slot (its neighbour plane)
    auto mirror_plane = [&](int kk, int zs) {
        const int gs = mod2(kk), kind = d.kind[zs];
        for (int t = tid; t < NP * GY; t += NT) {
            const int r = t / NP, p = t % NP;
#pragma unroll
            for (int q = 0; q < 5; ++q)
#pragma unroll
                for (int dir = 0; dir < 3; ++dir) {
                    const f2 g = sm.g[gs ^ 1][q * 3 + dir][r][p];
                    const float s = grad_flips(kind, 2, q, dir) ? -1.0f : 1.0f;
                    sm.g[gs][q * 3 + dir][r][p] = g * splat(s);
                }
        }
    };
    auto grad_plane = [&](int kk) {
        const int gs = mod2(kk);
        if (!zper && kk == nz) {
            mirror_plane(kk, 5);
            return;
        }
        const int vs = mod3(kk), vm = mod3(kk - 1), vp = mod3(kk + 1);
        const f2 izn = splat(sm.zline[9]), izm = splat(sm.zline[8]);
        for (int t = tid; t < NP * GY; t += NT) {
            const int gr = t / NP, p = t - gr * NP;
            int r = gr + 1, ym = -1;
            if (!yper) {  // a wall ghost row takes its partner's gradient, mirrored
                if (j0 - 2 + r == -1) ym = 2;
                if (j0 - 2 + r == ny) ym = 3;
                r += ym == 2 ? 1 : (ym == 3 ? -1 : 0);
            }
            // neighbours of the ring's outer columns are not read by any face
            const int wp = max(p - 1, 0), ep = min(p + 1, NP - 1);
            const float i0w = sm.xisn[max(2 * p - 1, 0)], i1 = sm.xisn[2 * p], i2 = sm.xisn[2 * p + 1];
            const f2 iyn = splat(sm.yisn[r]), iym = splat(sm.yisn[r - 1]);
#pragma unroll
            for (int q = 0; q < 5; ++q) {
                const f2 c = sm.v[vs][q][r][p];
                const float w = sm.v[vs][q][r][wp].y, e = sm.v[vs][q][r][ep].x;
                const float d1 = (c.y - c.x) * i1;
                f2 gx = {fmaf(c.x - w, i0w, d1), fmaf(e - c.y, i2, d1)};
                f2 gy = vfma(sm.v[vs][q][r + 1][p] - c, iyn, (c - sm.v[vs][q][r - 1][p]) * iym);
                f2 gz = vfma(sm.v[vp][q][r][p] - c, izn, (c - sm.v[vm][q][r][p]) * izm);
                if (ym >= 0) {
                    const int kind = d.kind[ym];
                    if (grad_flips(kind, 1, q, 0)) gx = vtraits<f2>::neg(gx);
                    if (grad_flips(kind, 1, q, 1)) gy = vtraits<f2>::neg(gy);
                    if (grad_flips(kind, 1, q, 2)) gz = vtraits<f2>::neg(gz);
                }
                sm.g[gs][q * 3 + 0][gr][p] = gx;
                sm.g[gs][q * 3 + 1][gr][p] = gy;
                sm.g[gs][q * 3 + 2][gr][p] = gz;
            }
        }
    };

    int ks_, zsm;
    resolve_1d(k0 - 1, nz, zper, 4, 5, ks_, zsm);
    const bool below_is_wall = zsm >= 0;
    __syncthreads();  // the ghost rules
    fetch(k0 - 2);
    const int gi = i0 + 2 * px, gj = j0 + ty;
    const bool mine = gi < nx && gj < ny, both = gi + 1 < nx, last = px == PX - 1;
    const float dtc = d.f_dt, bgd = d.f_beta_g * dtc, Tr = d.f_T_ref;
    const float fo[3] = {d.f_force[0] * dtc, d.f_force[1] * dtc, d.f_force[2] * dtc};
    const int g_axis = d.g_axis;
    // this thread's entry of Smem3P::zline
    auto zentry = [&](int k) {
        if (tid < 8) return reinterpret_cast<const float*>(zl + max(k + 1, 0))[tid];
        return tid == 8 ? zc[k + 2].is_next : (tid == 9 ? zc[k + 3].is_next : zc[k + 2].dt_w);
    };
    float zpre = tid < 11 ? zentry(k0 - 2) : 0.0f;
    f2 Fd[5] = {splat(0.0f), splat(0.0f), splat(0.0f), splat(0.0f), splat(0.0f)};
    float s0 = 0.0f, s1 = 0.0f, s2 = 0.0f, s3 = 0.0f;
    bool bad = false;
    // Iterations below k0 fill the pipeline: k0 - 4 .. k0 - 2 store planes
    // k0 - 2 .. k0, k0 - 2 makes the gradients of k0 - 1, k0 - 1 those of k0
    // and the z-faces below plane k0.
#pragma unroll 1
    for (int k = k0 - 4; k < k1; ++k) {
        store(k + 2);
        if (k >= k0 - 2) {
            if (tid < 11) {
                sm.zline[tid] = zpre;
                if (k + 1 < k1) zpre = zentry(k + 1);
            }
            __syncthreads();
            if (k > k0 - 2 || !below_is_wall) grad_plane(k + 1);
            __syncthreads();
        }
        if (k == k0 - 1 && below_is_wall) {
            mirror_plane(k0 - 1, zsm);
            __syncthreads();
        }
        const int vs = mod3(k), gs = mod2(k);
        f2 div[5];  // sum over the axes of dt / width * (flux out - flux in)
        if (k >= k0 - 1) {  // z-faces between planes k and k + 1
            CellNT3<f2> L, R;
            take_pair<2>(sm, vs, gs, ty + 2, px + 1, L);
            take_pair<2>(sm, mod3(k + 1), mod2(k + 1), ty + 2, px + 1, R);
            const int s = zper ? -1 : (k + 1 == 0 ? 4 : (k + 1 == nz ? 5 : -1));
            f2 F[5];
            face_pair<2, SCH>(L, R, Tz2,
                              rtlbfs::splat_line(*reinterpret_cast<const FaceLine<float>*>(sm.zline)),
                              [&](f2& mn, f2& m1, f2& m2, f2 rho) {
                                  if (s >= 0) {
                                      mn = splat(0.0f);
                                      m1 = rho * splat(d.f_bcU[s][0]);
                                      m2 = rho * splat(d.f_bcU[s][1]);
                                  }
                              },
                              F);
            const f2 az = splat(sm.zline[10]);
#pragma unroll
            for (int q = 0; q < 5; ++q) {
                div[q] = az * (F[q] - Fd[q]);
                Fd[q] = F[q];
            }
        }
        f2 dx[5];  // F east - F west; .y of the tile's last pair: F between a and b
        if (k >= k0) {
#pragma unroll 1
            for (int it = 0; it < 2; ++it) {  // y-faces below a and b; the tile's north row
                const int row = it ? TY : ty, p = it ? lane : px;
                if (it && (warp != NT / 32 - 1 || lane >= PX)) continue;
                CellNT3<f2> L, R;
                take_pair<1>(sm, vs, gs, row + 1, p + 1, L);
                take_pair<1>(sm, vs, gs, row + 2, p + 1, R);
                const int g = j0 + row;
                f2 F[5];
                face_pair<1, SCH>(L, R, Tz2, rtlbfs::splat_line(sm.yl[row]),
                                  [&](f2& mn, f2& m1, f2& m2, f2 rho) {
                                      if (yper) return;
                                      const int s = g == 0 ? 2 : (g == ny ? 3 : -1);
                                      if (s >= 0) {
                                          mn = splat(0.0f);
                                          m1 = rho * splat(d.f_bcU[s][2]);
                                          m2 = rho * splat(d.f_bcU[s][0]);
                                      }
                                  },
                                  F);
#pragma unroll
                for (int q = 0; q < 5; ++q) sm.fy[q][row][p] = F[q];
            }
            f2 F[5];
#pragma unroll 1
            for (int it = 1; it >= 0; --it) {  // the tile's east column; x-faces west of a and between a and b
                const int row = it ? lane : ty, p = it ? PX : px;
                if (it && (warp != 0 || lane >= TY)) continue;
                CellNT3<f2> L, R;
                take_pair<0>(sm, vs, gs, row + 2, p + 1, R);
                take_pair<0>(sm, vs, gs, row + 2, p, L);  // the pair to the west: its b, then a
#pragma unroll
                for (int q = 0; q < 5; ++q) {
                    L.q[q] = {L.q[q].y, R.q[q].x};
                    L.gn[q] = {L.gn[q].y, R.gn[q].x};
                    L.g1[q] = {L.g1[q].y, R.g1[q].x};
                    L.g2[q] = {L.g2[q].y, R.g2[q].x};
                }
                const FaceLine<f2> fl = {sm.xl[0][p], sm.xl[1][p], sm.xl[2][p], sm.xl[3][p],
                                         sm.xl[4][p], sm.xl[5][p], sm.xl[6][p], splat(0.0f)};
                const int g = i0 + 2 * p;
                face_pair<0, SCH>(L, R, Tz2, fl,
                                  [&](f2& mn, f2& m1, f2& m2, f2 rho) {
                                      if (xper) return;
                                      if (g == 0 || g == nx) {
                                          const int s = g == 0 ? 0 : 1;
                                          mn.x = 0.0f;
                                          m1.x = rho.x * d.f_bcU[s][1];
                                          m2.x = rho.x * d.f_bcU[s][2];
                                      }
                                      if (g + 1 == nx) {
                                          mn.y = 0.0f;
                                          m1.y = rho.y * d.f_bcU[1][1];
                                          m2.y = rho.y * d.f_bcU[1][2];
                                      }
                                  },
                                  F);
                // a gradient of the ring's outermost column, which no face reads
                if (it)
#pragma unroll
                    for (int q = 0; q < 5; ++q) sm.g[gs][q][row + 1][0].x = F[q].x;
            }
#pragma unroll
            for (int q = 0; q < 5; ++q) {
                const float e = __shfl_down_sync(0xffffffffu, F[q].x, 1);
                dx[q] = {F[q].y - F[q].x, last ? F[q].y : e - F[q].y};
            }
        }
        if (k + 3 <= k1 + 1) fetch(k + 3);  // in flight during the update
        const long long off = (long long)k * plane + (long long)gj * nx + gi;
        Rec qa = {0, 0, 0, 0}, qb = qa;
        int qTa = 0, qTb = 0;
        if (k >= k0 && mine) {  // the stored cells the update adds its increments to
            qa = rin[off];
            qTa = tin[off];
            if (both) {
                qb = rin[off + 1];
                qTb = tin[off + 1];
            }
        }
        f2 c0[5];  // before the barrier: the next plane takes this slot after it
#pragma unroll
        for (int q = 0; q < 5; ++q) c0[q] = sm.v[vs][q][ty + 2][px + 1];
        if (k >= k0 - 1) __syncthreads();
        if (k >= k0 && mine) {
            const f2 ax = {sm.xdtw[2 * px + 2], sm.xdtw[2 * px + 3]}, ay = splat(sm.ydtw[ty + 2]);
#pragma unroll
            for (int q = 0; q < 5; ++q) {
                if (last) dx[q].y = sm.g[gs][q][ty + 1][0].x - dx[q].y;
                div[q] = vfma(ax, dx[q], vfma(ay, sm.fy[q][ty + 1][px] - sm.fy[q][ty][px], div[q]));
            }
            const f2 dr = c0[0], T = Tz2 + c0[4];
            const f2 rho = splat(1.0f) + dr;
            const f2 buoy = splat(bgd) * (T - splat(Tr));
            const f2 inv = vtraits<f2>::rcp(rho - div[0]);
            f2 du[3], u1[3];
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                const f2 acc = a == g_axis ? buoy + splat(fo[a]) : splat(fo[a]);
                du[a] = (vfma(c0[1 + a], div[0], rho * acc) - div[1 + a]) * inv;
                u1[a] = c0[1 + a] + du[a];
            }
            const f2 dT = (T * div[0] - div[4]) * inv;
            const f2 T1 = T + dT, dr1 = dr - div[0];
            rout[off] = {P::add(qa.x, -div[0].x, 0), P::add(qa.y, du[0].x, 1),
                         P::add(qa.z, du[1].x, 1), P::add(qa.w, du[2].x, 1)};
            tout[off] = P::add(qTa, dT.x, 3);
            bad = bad || !(P::in_range(dr1.x, 0) && P::in_range(u1[0].x, 1) &&
                           P::in_range(u1[1].x, 1) && P::in_range(u1[2].x, 1) && P::in_range(T1.x, 3));
            const f2 q0 = vfma(c0[1], c0[1], vfma(c0[2], c0[2], c0[3] * c0[3]));
            const f2 q1 = vfma(u1[0], u1[0], vfma(u1[1], u1[1], u1[2] * u1[2]));
            const f2 den = f2{P::fsqrt(q0.x), P::fsqrt(q0.y)} + f2{P::fsqrt(q1.x), P::fsqrt(q1.y)};
            const f2 num = vfma(du[0], c0[1] + u1[0], vfma(du[1], c0[2] + u1[1], du[2] * (c0[3] + u1[2])));
            f2 dm = {den.x > 0.0f ? num.x * P::rcp(den.x) : 0.0f,
                     den.y > 0.0f ? num.y * P::rcp(den.y) : 0.0f};
            f2 e1 = q1, e2 = dT, e3 = T1;
            if (both) {
                rout[off + 1] = {P::add(qb.x, -div[0].y, 0), P::add(qb.y, du[0].y, 1),
                                 P::add(qb.z, du[1].y, 1), P::add(qb.w, du[2].y, 1)};
                tout[off + 1] = P::add(qTb, dT.y, 3);
                bad = bad || !(P::in_range(dr1.y, 0) && P::in_range(u1[0].y, 1) &&
                               P::in_range(u1[1].y, 1) && P::in_range(u1[2].y, 1) && P::in_range(T1.y, 3));
            } else {
                dm.y = e1.y = e2.y = e3.y = 0.0f;
            }
            s0 = fmaf(dm.x, dm.x, fmaf(dm.y, dm.y, s0));
            s1 += e1.x + e1.y;
            s2 = fmaf(e2.x, e2.x, fmaf(e2.y, e2.y, s2));
            s3 = fmaf(e3.x, e3.x, fmaf(e3.y, e3.y, s3));
        }
    }
    // residual sums: warp sums in the working precision, warps and units in FP64
    const float sum = rtlbfs::warp_sum4(bad ? NAN : s0, s1, s2, s3);
    __syncthreads();  // red lies over the fluxes
    if ((tid & 7) == 0) sm.red[warp][lane >> 3] = (double)sum;
    __syncthreads();
    rtlbfs::add_sums(sm.red, NT / 32, run->acc[slot3]);  // the next launch tests them
}

}  // namespace rtlbfs3
