// Row kernel of the CDI step: a 16-byte vector of cells per thread, any row length (nx).
//
// A block owns an x-y tile of W x TY cells (W = 16 vectors of 16 bytes) and marches along
// z, one barrier per plane.  Own warp w holds rows 2w and 2w + 1 of the tile, one vector of
// VX cells per thread; the last warp evaluates the sharpening ring (s_y of the rows below and
// above the tile, s_x of the columns left and right of it) and copies the halos.
//
// What bounded the kernel before (each plane of phi read twice from shared memory, 23 shared
// loads per vector and plane): the shared-memory data pipe, 71% of its cycles busy with a
// third of them bank conflicts of the scalar x-neighbour loads, and 26 integer instructions
// per cell of slot and address arithmetic.  So here
//   - what a thread reads of phi around its group stays in registers from the sharpening at
//     plane k+1 to the update at plane k+1 one iteration later (the group, its y and x
//     neighbours, its s_x, s_z): 14 shared loads per vector and plane;
//   - every staged array has the same row pitch and the plane loop is unrolled over the four
//     ring slots, so a shared access is one base register and an immediate;
//   - 14 rows and one ring warp make a block of 8 warps, two of which per SM leave each
//     thread 128 registers (10 warps per block left it 96, and the carried values spilled).
// FP32, aligned rows: 102.5 -> 82.3 instructions per cell; 256^3 72.4 -> 57.4 us per step of a
// run (4.63 -> 5.84 TB/s), 512^3 516 -> 420 us (5.20 -> 6.39 TB/s).
//
//   A = VX  (AL) rows start on 16-byte boundaries (nx % VX == 0): 16-byte cp.async and stores.
//   A = 1, 2    rows start at any element, or on pairs (FP32, nx even): a warp copies its rows
//               an element or a pair at a time (a lane
//               per column: contiguous runs) and stores element by element (through shared
//               memory, for contiguous stores: 89.1 against 86.4 us at 255^3 with the
//               14-row tile).  255^3 FP32:
//               139 us with one cell per thread (32x8 tile) -> 83.6 us; 385^3 501 -> 308 us; 254^3 by
//               pairs 135 -> 76.9 us, RK4 at 254^3 456 (by elements) -> 376 us.
// The arithmetic is that of every other forward kernel, in the same order: the fields are the
// same bit for bit.
#pragma once

#include "cdi_async.cuh"
#include "cdi_fwd_common.cuh"
#include "cdi_reduce.cuh"
#include "cdi_row.cuh"

namespace cdi {

template <typename T, int TY, bool RK, int NV>
struct RowCfg : RowGeo<T, TY> {
    using G = RowGeo<T, TY>;
    static constexpr int NVS = NV;            // velocity slots
    static constexpr int OVEL = G::NS * G::PHI, OSX = OVEL + NVS * G::VEL, OSY = OSX + 2 * G::SXS;
    static constexpr int RKO = G::H * G::W;   // a plane of one Runge-Kutta operand (RK: two operands, two slots)
    static constexpr int ORK = OSY + 2 * G::SYS;
    static constexpr size_t bytes = sizeof(T) * (size_t)(ORK + (RK ? 4 * RKO : 0));
    static_assert(G::VEL >= G::PHI, "the prologue's first phi plane borrows a velocity slot");
};

template <typename T, int TY, bool RK, bool ZR, int A, int NV>
__global__ void __launch_bounds__(RowCfg<T, TY, RK, NV>::NT, 512 / RowCfg<T, TY, RK, NV>::NT)
fwd_row_kernel(const FwdArgs<T> a, const int nchunks, const int chained)
{
    using C = RowCfg<T, TY, RK, NV>;
    using VV = V16<T>;
    constexpr int VX = C::VX, W = C::W, H = C::H, PP = C::PP, TX = C::TX;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T *const sm = reinterpret_cast<T *>(smem_raw);

    const int tid = threadIdx.x;
    const int nx = a.nx, ny = a.ny, nz = a.nz;
    const long long plane = (long long)nx * ny;
    const int tiles_x = (nx + W - 1) / W;
    const int ntiles = tiles_x * ((ny + H - 1) / H);
    const T c_adv = a.c.c_adv, c_dif = a.c.c_dif, c_shp = a.c.c_shp, c_upd = a.c.c_upd;
    unsigned *const st = a.red.status;
    (void)st;

    const bool is_own = tid < C::NOWN;
    const int lane = tid & 31, tx = tid % TX;
    // the row of this thread's group: own 0..H-1; the ring warp's -1 and H
    const int ty = is_own ? tid / TX : (lane < TX ? -1 : H);
    const bool has_xr = (lane & 15) < TY;  // ring warp: an x-ring cell, row lane & 15, left or right
    // the group's place: phi row ty + d of slot S at bp[S PHI + (1 + d) PP], u / w row ty at
    // bp[.. - PP], v row ty at bp[.. + VO] (row ty - 1 one pitch below), s_x row ty at
    // bp[.. - PP], s_y row ty at bp[..]; xb: the same for the x-ring cell
    T *const bp = sm + (ty + 1) * PP + VX + tx * VX;
    T *const xb = sm + ((lane & 15) + 1) * PP + VX + (lane < 16 ? -1 : W);
    constexpr bool AL = A == VX;
    RowStage<T, TY, A> cp(sm, tid, ty, tx);

    // Sharpening of the group's cells c, from its y neighbours, the planes below (zn) and
    // above (zp) and the x neighbours L, R.
    auto sharp = [&](const T *c, const T *yn, const T *yp, const T *zn, const T *zp, T L, T R, T *s0, T *s1, T *s2) {
#pragma unroll
        for (int i = 0; i < VX; ++i) {
            const T g0 = (i + 1 < VX ? c[i + 1] : R) - (i > 0 ? c[i - 1] : L);
            const T g1 = yp[i] - yn[i];
            const T g2 = zp[i] - zn[i];
            const T q = fma(g2, g2, fma(g1, g1, fma(g0, g0, NumLim<T>::tiny())));
            const T inv = rsqrt_t(q);
            const T wgt = c[i] * (T(1) - c[i]) * inv;
            s0[i] = wgt * g0;
            s1[i] = wgt * g1;
            s2[i] = wgt * g2;
        }
    };
    // s_x of the x-ring cell at phi offset o of its plane, pn / pp the cell in the planes below
    // and above
    auto sharp_cell = [&](const T *o, T p, T pn, T pp) {
        const T g0 = o[1] - o[-1];
        const T g1 = o[PP] - o[-PP];
        const T g2 = pp - pn;
        const T q = fma(g2, g2, fma(g1, g1, fma(g0, g0, NumLim<T>::tiny())));
        const T inv = rsqrt_t(q);
        return p * (T(1) - p) * inv * g0;
    };

    const unsigned rkb = cp.own_base(sm, ty, tx);
    (void)rkb;

    Acc<T> acc;
    acc.init();
    // The record is the last Runge-Kutta stage's, which overwrites the others': they skip it.
    const bool stats = !RK || a.red.update_run;
    bool dep_waited = !chained;  // the previous grid on the stream has completed
    if (!chained) grid_dep_wait();

    const int zlo = ZR ? a.z_lo : 0, zr = ZR ? a.z_hi - a.z_lo : nz;
    UnitIter<W, H> units(ntiles, zr, nchunks);
    Unit un;
    while (units.next(un, ntiles, tiles_x, zr, nchunks)) {
        const int x0 = un.x0, y0 = un.y0, z0 = un.z0 + zlo, z1 = un.z1 + zlo;

        cp.plan(sm, x0, y0, ty, tx, nx, ny, plane, st);
        auto issue_vel = [&](long long zo, auto SO) {
            cp.template vel<decltype(SO)::value>(a.u + zo, a.v + zo, a.w + zo);
        };
        // Runge-Kutta stage operands of plane zo into slot B: staged a plane ahead rather than
        // held in registers across the sharpening (which spilled 88 bytes per thread).
        auto issue_rk = [&](long long zo, auto B) {
            constexpr int so = C::ORK + decltype(B)::value * 2 * C::RKO;
            if (!is_own) return;
            if (a.rk_base) cp.template own<so>(rkb, a.rk_base + zo);
            if (a.rk_q) cp.template own<so + C::RKO>(rkb, a.rk_q + zo);
        };

        // Slot of plane z, phi and velocities: (z - z0) mod 4.
        __syncthreads();  // the previous unit's readers are done with every slot
        // The face velocities are never written by a step: staged (and the w below
        // plane z0 loaded) before waiting for the previous grid on the stream if that is one
        // of the same call (chained).
        long long zo = (long long)CDI_CHK(z0, nz, st) * plane;  // element offset of plane k
        issue_vel(zo, IC<C::OVEL>{});
        const int own_x = x0 + tx * VX, own_y = y0 + ty;
        const int nown = is_own && own_y < ny ? min(VX, nx - own_x) : 0;  // own cells inside the box (<= 0: none)
        T wlo[VX];  // w on the face below plane z0 (own cells)
        if (is_own) {
            const T *src = a.w + (long long)wrapi(z0 - 1, nz) * plane;
            if constexpr (AL) {
                VV::ld(wlo, src + cp.g[0]);
            } else {
                const int yo = wrapi(own_y, ny) * nx;
#pragma unroll
                for (int i = 0; i < VX; ++i)
                    wlo[i] = __ldg(src + CDI_CHK(yo + (i < nown ? own_x + i : 0), plane, st));
            }
        }
        if (!dep_waited) {
            grid_dep_wait();
            dep_waited = true;
        }
        int zq = wrapi(z0 - 2, nz);  // wrapped index of the next phi plane to stage
        auto next_phi = [&](auto SO) {
            cp.template halo2<decltype(SO)::value>(a.phi + (long long)CDI_CHK(zq, nz, st) * plane);
            zq = zq + 1 == nz ? 0 : zq + 1;
        };
        // planes z0-2 (in the velocity slot of plane z0+3, free until then), z0-1 .. z0+2
        constexpr int M2 = C::OVEL + (C::NVS - 1) * C::VEL;
        next_phi(IC<M2>{});
        next_phi(IC<3 * C::PHI>{});
        next_phi(IC<0>{});
        next_phi(IC<C::PHI>{});
        next_phi(IC<2 * C::PHI>{});
        if constexpr (RK) issue_rk(zo, IC<0>{});
        cp_async_commit();
        if constexpr (C::NVS == 4) {
            if (z0 + 1 < z1) issue_vel(zo + plane, IC<C::OVEL + C::VEL>{});
            if (z0 + 2 < z1) issue_vel(zo + 2 * plane, IC<C::OVEL + 2 * C::VEL>{});
        }
        cp_async_commit();
        cp_async_wait<1>();
        __syncthreads();

        // Prologue: s_z at plane z0-1 (own), s at plane z0 (own + ring), flux at z0-1/2.
        // Carried: cK, ynK, ypK, LK, RK phi around the group at plane k; cN the group at plane
        // k+1; sxK, szK its s_x, s_z at plane k; Fzm the flux through its lower z faces.  The
        // x-ring cell's phi at planes k, k+1: pK, pN.
        T cK[VX], cN[VX], ynK[VX], ypK[VX], LK, RK_, sxK[VX], szK[VX], Fzm[VX], pK = T(0), pN = T(0);
        {
            const T *P0 = bp + PP;                        // plane z0
            const T *Pm1 = P0 + 3 * C::PHI, *Pm2 = P0 + M2, *P1 = P0 + C::PHI;
            VV::ld(cK, P0);
            VV::ld(ynK, P0 - PP);
            VV::ld(ypK, P0 + PP);
            VV::ld(cN, P1);
            LK = P0[-1];
            RK_ = P0[VX];
            T cm[VX], s1[VX];
            VV::ld(cm, Pm1);
            sharp(cK, ynK, ypK, cm, cN, LK, RK_, sxK, s1, szK);
            VV::st(bp + C::OSY, s1);
            if (is_own) {
                VV::st(bp + C::OSX - PP, sxK);
                T ym[VX], yq[VX], zm[VX], a0[VX], a1[VX], szm[VX];
                VV::ld(ym, Pm1 - PP);
                VV::ld(yq, Pm1 + PP);
                VV::ld(zm, Pm2);
                sharp(cm, ym, yq, zm, cK, Pm1[-1], Pm1[VX], a0, a1, szm);
#pragma unroll
                for (int i = 0; i < VX; ++i)
                    Fzm[i] = flux(c_adv * wlo[i], c_dif, c_shp, cm[i], cK[i], szm[i], szK[i]);
            } else if (has_xr) {
                const T *x = xb + PP;
                pK = x[0];
                pN = x[C::PHI];
                xb[C::OSX - PP] = sharp_cell(x, pK, x[3 * C::PHI], pN);
            }
        }
        __syncthreads();  // the slots of planes z0-2 and z0-1 are free
        if (z0 + 3 <= z1 + 1) next_phi(IC<3 * C::PHI>{});
        cp_async_commit();

        T *op = a.out + zo;  // plane k of the output
        const int go = nown > 0 ? own_y * nx + own_x : 0;
        // One plane: S = (k - z0) mod 4.
        auto body = [&](auto SC, const int k) {
            constexpr int S = decltype(SC)::value, S1 = (S + 1) & 3, S2 = (S + 2) & 3;
            constexpr int b = S & 1, b1 = b ^ 1;
            // S1: phi plane k+2 and the velocities of plane k have landed, and every thread
            // has left iteration k-1.
            cp_async_wait<1>();
            __syncthreads();
            if constexpr (RK || C::NVS == 2) {  // a group of its own, before plane k+4's: landed at the next barrier
                if (k + 1 < z1) {
                    if constexpr (RK) issue_rk(zo + plane, IC<b1>{});
                    if constexpr (C::NVS == 2) issue_vel(zo + plane, IC<C::OVEL + b1 * C::VEL>{});
                }
                cp_async_commit();
            }
            if (k + 4 <= z1 + 1) next_phi(IC<S * C::PHI>{});
            if constexpr (C::NVS == 4) {
                if (k + 3 < z1) issue_vel(zo + 3 * plane, IC<C::OVEL + ((S + 3) & 3) * C::VEL>{});
            }
            cp_async_commit();

            // B: sharpening at plane k+1 (every warp).
            T cP[VX], ynN[VX], ypN[VX], LN, RN, sxN[VX], szN[VX];
            {
                const T *P1 = bp + S1 * C::PHI + PP;
                VV::ld(cP, bp + S2 * C::PHI + PP);
                VV::ld(ynN, P1 - PP);
                VV::ld(ypN, P1 + PP);
                LN = P1[-1];
                RN = P1[VX];
                T s1[VX];
                sharp(cN, ynN, ypN, cK, cP, LN, RN, sxN, s1, szN);
                VV::st(bp + C::OSY + b1 * C::SYS, s1);
            }
            // No barrier here: phase C reads only the s_x, s_y of plane k, which were written
            // before S1, and the own s_x, s_z of plane k+1 from registers.
            if (!is_own) {
                if (has_xr) {
                    const T pP = xb[S2 * C::PHI + PP];
                    xb[C::OSX + b1 * C::SXS - PP] = sharp_cell(xb + S1 * C::PHI + PP, pN, pK, pP);
                    pK = pN;
                    pN = pP;
                }
            } else {
                VV::st(bp + C::OSX + b1 * C::SXS - PP, sxN);
                // C: fluxes and update at plane k (x and y faces telescoped, the z face
                // below carried).
                const T *sx = bp + C::OSX + b * C::SXS - PP, *sy = bp + C::OSY + b * C::SYS;
                T *const vel = bp + C::OVEL + (S & (C::NVS - 1)) * C::VEL;
                T syn[VX], syp[VX], uc[VX], vc[VX], vn[VX], wc[VX];
                VV::ld(syn, sy - PP);
                VV::ld(syp, sy + PP);
                VV::ld(uc, vel - PP);
                VV::ld(vc, vel + C::VO);
                VV::ld(vn, vel + C::VO - PP);
                VV::ld(wc, vel + C::WO - PP);
                const T sxL = sx[-1], sxR = sx[VX];
                const T uL = vel[-PP - 1];
                T o[VX];
#pragma unroll
                for (int i = 0; i < VX; ++i) {
                    const T xl = i > 0 ? cK[i - 1] : LK, xr = i + 1 < VX ? cK[i + 1] : RK_;
                    const T ul = i > 0 ? uc[i - 1] : uL;
                    const T sl = i > 0 ? sxK[i - 1] : sxL, sr = i + 1 < VX ? sxK[i + 1] : sxR;
                    T adv = uc[i] * (cK[i] + xr);
                    adv = fma(-ul, xl + cK[i], adv);
                    adv = fma(vc[i], cK[i] + ypK[i], adv);
                    adv = fma(-vn[i], ynK[i] + cK[i], adv);
                    const T dif = fma(T(-4), cK[i], (xl + xr) + (ynK[i] + ypK[i]));
                    const T shp = (sr - sl) + (syp[i] - syn[i]);
                    const T Fzp = flux(c_adv * wc[i], c_dif, c_shp, cK[i], cN[i], szK[i], szN[i]);
                    const T div = fma(c_adv, adv, fma(-c_dif, dif, fma(c_shp, shp, Fzp - Fzm[i])));
                    if constexpr (RK) o[i] = -c_upd * div;  // r = dt * RHS, combined below
                    else o[i] = fma(-c_upd, div, cK[i]);
                    Fzm[i] = Fzp;
                }
                if constexpr (RK) {
                    if (nown > 0) {
                        T *const qout = a.rk_qout ? a.rk_qout + (zo + go) : nullptr;
                        const T *const ro = sm + C::ORK + b * 2 * C::RKO + ty * W + tx * VX;
                        T qo[VX], rb[VX], rq[VX];
                        VV::ld(rb, ro);  // (unused values where there is no such operand)
                        VV::ld(rq, ro + C::RKO);
#pragma unroll
                        for (int i = 0; i < VX; ++i) {
                            const T r = o[i];
                            const T base = a.rk_base ? rb[i] : cK[i];
                            const T q = a.rk_q ? rq[i] : T(0);
                            o[i] = fma(a.rk_delta, q, fma(a.rk_alpha, r, base));
                            qo[i] = fma(a.rk_beta, r, a.rk_mu * (a.rk_q ? q : cK[i]));
                        }
                        if (qout) {
                            if constexpr (AL) {
                                VV::st(qout, qo);
                            } else {
                                store_cells<A, VX>(qout, qo, nown);
                            }
                        }
                    }
                }
                if constexpr (AL) {
                    if (nown > 0) {
                        VV::st(op + cp.g[0], o);
                        if (stats) acc.template add_group<VX>(o, a.c.tol);
                    }
                } else {
                    if (stats && nown > 0) acc.template add_group_n<VX>(o, nown, a.c.tol);
                    store_cells<A, VX>(op + go, o, nown);
                }
            }
#pragma unroll
            for (int i = 0; i < VX; ++i) {
                cK[i] = cN[i];
                cN[i] = cP[i];
                ynK[i] = ynN[i];
                ypK[i] = ypN[i];
                sxK[i] = sxN[i];
                szK[i] = szN[i];
            }
            LK = LN;
            RK_ = RN;
            zo += plane;
            op += plane;
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
    grid_dep_launch();  // the next step may start staging its velocities
    if (stats) reduce_and_finish<ZR>(acc, a.red);
}

}  // namespace cdi
