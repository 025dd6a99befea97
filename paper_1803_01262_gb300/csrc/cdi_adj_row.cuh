// Row kernel of the adjoint step: the structure of the forward row kernel (cdi_fwd_row.cuh) for
// the formulas of cdi_adj.cu, any row length.  phi and lam' travel in two rings of four slots;
// what a thread reads around its vector it carries in registers from gbar at plane k+1 to the
// update at plane k+1.  The formulas are arranged for fewer operations than the per-cell
// kernel's, with raw differences dl of lam':
//   gd = g . dl,  r = gd / m,  gbar = c p (1 - p) / m (dl - g r / m),  local term (1 - 2 p) c r,
// c = gamma dt / (2 dx) (sbar = c dl), and dt / dx folded into the face coefficients.  What of a
// plane's update is known one plane earlier (local term, lower z face, gbar_z below) is carried as
// one sum: carried apart, the three spilled.
//
// FP32, aligned rows: 148 -> 105 instructions per cell; 256^3 100.5 -> 83.5 us per step (4.0 -> 4.8
// TB/s), with velocity gradients 156 -> 142 us (5.7 TB/s); FP64 128^3 348 -> 316 us (fewer FP64
// operations).  Other rows, against one cell per thread: 255^3 FP32 172.5 -> 106 us, with
// gradients 322 -> 171 us; 254^3 (rows on pairs) 171 -> 100 and 315 -> 139; FP64 129^3 609 -> 384 us.
#pragma once

#include "cdi_row.cuh"

namespace cdi {

template <typename T, int TY, int A>
struct AdjRowCfg : RowGeo<T, TY> {
    using G = RowGeo<T, TY>;
    // velocity slots; other rows: two, which leaves L1 32 kB more (255^3 FP32 121 -> 106 us, with
    // gradients 209 -> 192)
    static constexpr int NVS = A == G::VX ? 4 : 2;
    static constexpr int OLAM = G::NS * G::PHI, OVEL = 2 * G::NS * G::PHI;
    static constexpr int OGX = OVEL + NVS * G::VEL, OGY = OGX + 2 * G::SXS;
    static constexpr size_t bytes = sizeof(T) * (size_t)(OGY + 2 * G::SYS);
    static_assert(G::VEL >= 2 * G::PHI, "the prologue's first planes borrow a velocity slot");
};

// Add the group's n cells to memory by reductions at L2 (no other thread of the launch touches
// them): the sums come back to no register, so no load's latency sits at the end of a plane.
// With loads and stores instead, 256^3 FP32 with velocity gradients took 202 us, 142 us so.  Rows
// at any element: pairs where the address allows, for fewer reductions (255^3 192 -> 171 us; a
// neighbour's first cell fetched by a shuffle, so that every lane issues two, 168 but it spills).
template <int A>
__device__ __forceinline__ void red_add(float *p, const float *v, int n)
{
    if constexpr (A == 4) {
        asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(v[0]), "f"(v[1]), "f"(v[2]),
                     "f"(v[3])
                     : "memory");
    } else if constexpr (A == 2) {
#pragma unroll
        for (int i = 0; i < 4; i += 2)
            if (i < n)
                asm volatile("red.global.add.v2.f32 [%0], {%1, %2};" ::"l"(p + i), "f"(v[i]), "f"(v[i + 1]) : "memory");
    } else if (n == 4) {  // pairs where they lie on 8-byte boundaries
        const int o = ((size_t)p >> 2) & 1;
        if (o) atomicAdd(p, v[0]);
        asm volatile("red.global.add.v2.f32 [%0], {%1, %2};" ::"l"(p + o), "f"(o ? v[1] : v[0]), "f"(o ? v[2] : v[1])
                     : "memory");
        if (o) atomicAdd(p + 3, v[3]);
        else asm volatile("red.global.add.v2.f32 [%0], {%1, %2};" ::"l"(p + 2), "f"(v[2]), "f"(v[3]) : "memory");
    } else {
#pragma unroll
        for (int i = 0; i < 3; ++i)
            if (i < n) atomicAdd(p + i, v[i]);
    }
}
template <int A>
__device__ __forceinline__ void red_add(double *p, const double *v, int n)
{
#pragma unroll
    for (int i = 0; i < 2; ++i)
        if (A == 2 || i < n) atomicAdd(p + i, v[i]);
}

// VEL: the velocity gradients are accumulated (a.gu, a.gv, a.gw not null).
template <typename T, int TY, bool VEL, int A>
__global__ void __launch_bounds__(AdjRowCfg<T, TY, A>::NT, 512 / AdjRowCfg<T, TY, A>::NT)
adj_row_kernel(const AdjArgs<T> a, const int nchunks, const int chained)
{
    using C = AdjRowCfg<T, TY, A>;
    using VV = V16<T>;
    constexpr int VX = C::VX, W = C::W, H = C::H, PP = C::PP, TX = C::TX, PHI = C::PHI;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T *const sm = reinterpret_cast<T *>(smem_raw);

    const int tid = threadIdx.x;
    const int nx = a.nx, ny = a.ny, nz = a.nz;
    const long long plane = (long long)nx * ny;
    const int tiles_x = (nx + W - 1) / W;
    const int ntiles = tiles_x * ((ny + H - 1) / H);
    const T c_sb = a.c_shp_adj, cau = a.c.c_upd * a.c.c_adv, cdu = a.c.c_upd * a.c.c_dif;
    const T c_vel = a.c.c_upd * a.c_vel;
    unsigned *const st = a.status;
    (void)st;
    (void)c_vel;

    const bool is_own = tid < C::NOWN;
    const int lane = tid & 31, tx = tid % TX;
    const int ty = is_own ? tid / TX : (lane < TX ? -1 : H);  // the ring warp's rows -1 and H
    const bool has_xr = (lane & 15) < TY;                     // ring warp: an x-ring cell
    T *const bp = sm + (ty + 1) * PP + VX + tx * VX;
    T *const xb = sm + ((lane & 15) + 1) * PP + VX + (lane < 16 ? -1 : W);
    constexpr bool AL = A == VX;
    RowStage<T, TY, A> cp(sm, tid, ty, tx);

    // gbar (b0, b1, b2) and the local term of the group's cells p, from the phi differences g
    // and the lam' differences dl
    auto gbar1 = [&](T p, T g0, T g1, T g2, T d0, T d1, T d2, T &b0, T &b1, T &b2, T &tl) {
        const T inv = inv_norm(g0, g1, g2);
        const T gd = fma(g2, d2, fma(g1, d1, g0 * d0));
        const T r = gd * inv, t = r * inv, ci = c_sb * inv;
        const T wgt = p * (T(1) - p) * ci;
        b0 = wgt * fma(-g0, t, d0);
        b1 = wgt * fma(-g1, t, d1);
        b2 = wgt * fma(-g2, t, d2);
        tl = fma(T(-2), p, T(1)) * (c_sb * r);
    };
    auto gbar = [&](const T *c, const T *yn, const T *yp, const T *zn, const T *zp, T L, T R, const T *l, const T *lyn,
                    const T *lyp, const T *lzn, const T *lzp, T lL, T lR, T *b0, T *b1, T *b2, T *tl) {
#pragma unroll
        for (int i = 0; i < VX; ++i)
            gbar1(c[i], (i + 1 < VX ? c[i + 1] : R) - (i > 0 ? c[i - 1] : L), yp[i] - yn[i], zp[i] - zn[i],
                  (i + 1 < VX ? l[i + 1] : lR) - (i > 0 ? l[i - 1] : lL), lyp[i] - lyn[i], lzp[i] - lzn[i], b0[i],
                  b1[i], b2[i], tl[i]);
    };
    // gbar_x of the x-ring cell: o, q its places in phi and lam'; pn, pp, ln, lp the planes
    // below and above
    auto gbar_x = [&](const T *o, T p, T pn, T pp, const T *q, T ln, T lp) {
        T b0, b1, b2, tl;
        gbar1(p, o[1] - o[-1], o[PP] - o[-PP], pp - pn, q[1] - q[-1], q[PP] - q[-PP], lp - ln, b0, b1, b2, tl);
        return b0;
    };

    bool dep_waited = !chained;  // the previous grid on the stream has completed
    if (!chained) grid_dep_wait();
    UnitIter<W, H> units(ntiles, nz, nchunks);
    Unit un;
    while (units.next(un, ntiles, tiles_x, nz, nchunks)) {
        const int x0 = un.x0, y0 = un.y0, z0 = un.z0, z1 = un.z1;
        cp.plan(sm, x0, y0, ty, tx, nx, ny, plane, st);
        auto issue_vel = [&](long long zo, auto SO) {
            cp.template vel<decltype(SO)::value>(a.u + zo, a.v + zo, a.w + zo);
        };

        // Slot of plane z in every ring: (z - z0) mod 4.  The velocities (and w below plane z0)
        // before waiting for the previous grid on the stream if that is one of the same call
        // (chained); phi, lam' and the accumulated
        // velocity gradients, which it may write, only after.
        __syncthreads();  // the previous unit's readers are done with every slot
        long long zo = (long long)CDI_CHK(z0, nz, st) * plane;  // element offset of plane k
        issue_vel(zo, IC<C::OVEL>{});
        const int own_x = x0 + tx * VX, own_y = y0 + ty;
        const int nown = is_own && own_y < ny ? min(VX, nx - own_x) : 0;  // own cells inside the box (<= 0: none)
        const int go = nown > 0 ? (int)CDI_CHK(own_y * nx + own_x, plane, st) : 0;
        T wlo[VX];  // w on the face below plane z0 (own cells)
        if (is_own) {
            const T *src = a.w + (long long)wrapi(z0 - 1, nz) * plane + go;
#pragma unroll
            for (int i = 0; i < VX; ++i) wlo[i] = __ldg(src + (i < nown ? i : 0));
        }
        if (!dep_waited) {
            grid_dep_wait();
            dep_waited = true;
        }
        int zq = wrapi(z0 - 2, nz);  // wrapped index of the next phi / lam' plane to stage
        auto next_planes = [&](auto SP, auto SL) {
            const long long o = (long long)CDI_CHK(zq, nz, st) * plane;
            cp.template halo2<decltype(SP)::value>(a.phi + o);
            cp.template halo2<decltype(SL)::value>(a.lam + o);
            zq = zq + 1 == nz ? 0 : zq + 1;
        };
        // planes z0-2 (in the velocity slot of plane z0+3, free until then), z0-1 .. z0+2
        constexpr int M2 = C::OVEL + (C::NVS - 1) * C::VEL;
        next_planes(IC<M2>{}, IC<M2 + PHI>{});
        next_planes(IC<3 * PHI>{}, IC<C::OLAM + 3 * PHI>{});
        next_planes(IC<0>{}, IC<C::OLAM>{});
        next_planes(IC<PHI>{}, IC<C::OLAM + PHI>{});
        next_planes(IC<2 * PHI>{}, IC<C::OLAM + 2 * PHI>{});
        cp_async_commit();
        if constexpr (C::NVS == 4) {
            if (z0 + 1 < z1) issue_vel(zo + plane, IC<C::OVEL + C::VEL>{});
            if (z0 + 2 < z1) issue_vel(zo + 2 * plane, IC<C::OVEL + 2 * C::VEL>{});
        }
        cp_async_commit();
        cp_async_wait<1>();
        __syncthreads();

        // Prologue: gbar_z at plane z0-1 (own); gbar and the local term at z0 (own + ring); the
        // z-face term at z0-1/2.  Carried: phi (c) and lam' (l) of the group at planes k and
        // k+1, lam' around it at plane k, its gbar_x and gbar_z at plane k, and acK the part of
        // the update of plane k known before plane k+1 is (the local term, the lower z face's
        // term and gbar_z at plane k-1); VEL: also phi right of and above it.
        T cK[VX], cN[VX], lK[VX], lN[VX], lynK[VX], lypK[VX], lLK, lRK, gxK[VX], gzK[VX], acK[VX];
        T ypK[VX], RK_ = T(0), pK = T(0), pN = T(0), qK = T(0), qN = T(0);  // p, q: the x-ring cell
        {
            const T *P0 = bp + PP, *Q0 = P0 + C::OLAM;    // plane z0 of phi and lam'
            T yn[VX], cm[VX], lm[VX], b1[VX];
            VV::ld(cK, P0);
            VV::ld(yn, P0 - PP);
            VV::ld(ypK, P0 + PP);
            VV::ld(cN, P0 + PHI);
            VV::ld(cm, P0 + 3 * PHI);
            VV::ld(lK, Q0);
            VV::ld(lynK, Q0 - PP);
            VV::ld(lypK, Q0 + PP);
            VV::ld(lN, Q0 + PHI);
            VV::ld(lm, Q0 + 3 * PHI);
            RK_ = P0[VX];
            lLK = Q0[-1];
            lRK = Q0[VX];
            gbar(cK, yn, ypK, cm, cN, P0[-1], RK_, lK, lynK, lypK, lm, lN, lLK, lRK, gxK, b1, gzK, acK);
            VV::st(bp + C::OGY, b1);
            if (is_own) {
                VV::st(bp + C::OGX - PP, gxK);
                const T *Pm = P0 + 3 * PHI, *Qm = Q0 + 3 * PHI;  // plane z0-1
                T y0_[VX], y1_[VX], z0_[VX], v0_[VX], v1_[VX], w0_[VX], a0[VX], a1[VX], gzm[VX], tt[VX];
                VV::ld(y0_, Pm - PP);
                VV::ld(y1_, Pm + PP);
                VV::ld(z0_, P0 + M2);
                VV::ld(v0_, Qm - PP);
                VV::ld(v1_, Qm + PP);
                VV::ld(w0_, P0 + M2 + PHI);
                gbar(cm, y0_, y1_, z0_, cK, Pm[-1], Pm[VX], lm, v0_, v1_, w0_, lK, Qm[-1], Qm[VX], a0, a1, gzm, tt);
#pragma unroll
                for (int i = 0; i < VX; ++i) acK[i] += fma(lK[i] - lm[i], fma(cau, wlo[i], -cdu), gzm[i]);
            } else if (has_xr) {
                const T *x = xb + PP, *y = x + C::OLAM;
                pK = x[0];
                pN = x[PHI];
                qK = y[0];
                qN = y[PHI];
                xb[C::OGX - PP] = gbar_x(x, pK, x[3 * PHI], pN, y, y[3 * PHI], qN);
            }
        }
        __syncthreads();  // the slots of planes z0-2 and z0-1 are free
        if (z0 + 3 <= z1 + 1) next_planes(IC<3 * PHI>{}, IC<C::OLAM + 3 * PHI>{});
        cp_async_commit();

        // One plane: S = (k - z0) mod 4.
        auto body = [&](auto SC, const int k) {
            constexpr int S = decltype(SC)::value, S1 = (S + 1) & 3, S2 = (S + 2) & 3;
            constexpr int b = S & 1, b1 = b ^ 1;
            // S1: planes k+2 and the velocities of plane k have landed, and every thread has
            // left iteration k-1.
            cp_async_wait<1>();
            __syncthreads();
            if constexpr (C::NVS == 2) {  // a group of its own: landed at the next barrier
                if (k + 1 < z1) issue_vel(zo + plane, IC<C::OVEL + b1 * C::VEL>{});
                cp_async_commit();
            }
            if (k + 4 <= z1 + 1) next_planes(IC<S * PHI>{}, IC<C::OLAM + S * PHI>{});
            if constexpr (C::NVS == 4) {
                if (k + 3 < z1) issue_vel(zo + 3 * plane, IC<C::OVEL + ((S + 3) & 3) * C::VEL>{});
            }
            cp_async_commit();
            if (!AL && !VEL && k + 5 < z1) {
                const long long zp = zo + 5 * plane;
                cp.ahead(a.u + zp);
                cp.ahead(a.v + zp);
                cp.ahead(a.w + zp);
                cp.ahead(a.phi + zp);
                cp.ahead(a.lam + zp);
            }

            // B: gbar at plane k+1 (every warp).
            T cP[VX], lP[VX], ypN[VX], RN, lynN[VX], lypN[VX], lLN, lRN, gxN[VX], gzN[VX], tN[VX];
            {
                const T *P1 = bp + S1 * PHI + PP, *Q1 = P1 + C::OLAM;
                T yn[VX], gy[VX];
                VV::ld(cP, bp + S2 * PHI + PP);
                VV::ld(yn, P1 - PP);
                VV::ld(ypN, P1 + PP);
                VV::ld(lP, bp + C::OLAM + S2 * PHI + PP);
                VV::ld(lynN, Q1 - PP);
                VV::ld(lypN, Q1 + PP);
                RN = P1[VX];
                lLN = Q1[-1];
                lRN = Q1[VX];
                gbar(cN, yn, ypN, cK, cP, P1[-1], RN, lN, lynN, lypN, lK, lP, lLN, lRN, gxN, gy, gzN, tN);
                VV::st(bp + C::OGY + b1 * C::SYS, gy);
            }
            // No barrier here: phase C reads only what was written before S1 (gbar_x of the
            // neighbours and gbar_y at plane k) and registers.
            if (!is_own) {
                if (has_xr) {
                    const T pP = xb[S2 * PHI + PP], qP = xb[C::OLAM + S2 * PHI + PP];
                    xb[C::OGX + b1 * C::SXS - PP] =
                        gbar_x(xb + S1 * PHI + PP, pN, pK, pP, xb + C::OLAM + S1 * PHI + PP, qK, qP);
                    pK = pN;
                    pN = pP;
                    qK = qN;
                    qN = qP;
                }
            } else {
                VV::st(bp + C::OGX + b1 * C::SXS - PP, gxN);
                // C: lam at plane k.
                const T *gx = bp + C::OGX + b * C::SXS - PP, *gy = bp + C::OGY + b * C::SYS;
                const T *vel = bp + C::OVEL + (S & (C::NVS - 1)) * C::VEL;
                T gyn[VX], gyp[VX], uc[VX], vc[VX], vn[VX], wc[VX];
                VV::ld(gyn, gy - PP);
                VV::ld(gyp, gy + PP);
                VV::ld(uc, vel - PP);
                VV::ld(vc, vel + C::VO);
                VV::ld(vn, vel + C::VO - PP);
                VV::ld(wc, vel + C::WO - PP);
                const T gxL = gx[-1], gxR = gx[VX], uL = vel[-PP - 1];
                T o[VX], dx[VX], dy[VX], dz[VX];
#pragma unroll
                for (int i = 0; i < VX; ++i) {
                    const T lc = lK[i];
                    const T ul = i > 0 ? uc[i - 1] : uL;
                    const T Dxm = i > 0 ? dx[i - 1] : lc - lLK;
                    const T Dym = lc - lynK[i];
                    dx[i] = (i + 1 < VX ? lK[i + 1] : lRK) - lc;
                    dy[i] = lypK[i] - lc;
                    dz[i] = lN[i] - lc;
                    T pb = fma(dx[i], fma(cau, uc[i], cdu), Dxm * fma(cau, ul, -cdu));
                    pb = fma(dy[i], fma(cau, vc[i], cdu), fma(Dym, fma(cau, vn[i], -cdu), pb));
                    pb = fma(dz[i], fma(cau, wc[i], cdu), pb);
                    const T gl = i > 0 ? gxK[i - 1] : gxL, gr = i + 1 < VX ? gxK[i + 1] : gxR;
                    pb += (gl - gr) + (gyn[i] - gyp[i]) + (acK[i] - gzN[i]);
                    o[i] = lc + pb;
                    acK[i] = fma(dz[i], fma(cau, wc[i], -cdu), tN[i] + gzK[i]);
                }
                if (nown > 0) {
                    const long long ko = (long long)CDI_CHK(k, nz, st) * plane + go;
                    if constexpr (AL) {
                        VV::st(a.out + ko, o);
                    } else {
                        store_cells<A, VX>(a.out + ko, o, nown);
                    }
                    if constexpr (VEL) {
                        T *const G3[3] = {a.gu + ko, a.gv + ko, a.gw + ko};
#pragma unroll
                        for (int q = 0; q < 3; ++q) {
                            T v[VX];
#pragma unroll
                            for (int i = 0; i < VX; ++i) {
                                const T pr = q == 0 ? (i + 1 < VX ? cK[i + 1] : RK_) : q == 1 ? ypK[i] : cN[i];
                                v[i] = (q == 0 ? dx[i] : q == 1 ? dy[i] : dz[i]) * c_vel * (cK[i] + pr);
                            }
                            red_add<A>(G3[q], v, nown);
                        }
                    }
                }
            }
#pragma unroll
            for (int i = 0; i < VX; ++i) {
                cK[i] = cN[i];
                cN[i] = cP[i];
                lK[i] = lN[i];
                lN[i] = lP[i];
                lynK[i] = lynN[i];
                lypK[i] = lypN[i];
                ypK[i] = ypN[i];
                gxK[i] = gxN[i];
                gzK[i] = gzN[i];
            }
            RK_ = RN;
            lLK = lLN;
            lRK = lRN;
            zo += plane;
        };
        for (int k = z0;;) {
            body(IC<0>{}, k);
            if (++k == z1) break;
            body(IC<1>{}, k);
            if (++k == z1) break;
            body(IC<2>{}, k);
            if (++k == z1) break;
            body(IC<3>{}, k);
            if (++k == z1) break;
        }
        cp_async_wait<0>();
    }
    if (!dep_waited) grid_dep_wait();
    grid_dep_launch();
}

}  // namespace cdi
