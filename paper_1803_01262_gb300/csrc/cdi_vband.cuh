// Vector row-band unit body of the batched CDI step, on the batch's padded copy
// of each box.
//
// The batch keeps its own copy of every box: each row of nx cells starts a row of
// pitch P = round_up(nx + 2, VX) elements (VX: a 16-byte vector), and the two
// positions after it hold its periodic continuation (cells 0 and 1).  Rows and planes
// then start on 16-byte boundaries whatever nx is, so a unit -- a band of whole rows
// [y0, y0 + hb) and a range of planes [z0, z1) -- is staged by 16-byte copies
// (each thread's few vectors of a region planned once per unit, rows outside [0, ny)
// wrapped in y) and one 4-byte copy for the cells left of x = 0 (a staged row has a
// vector of room there: pitch P + VX).  Each thread owns one group of VX consecutive
// cells of the band: whole rows, so no lane idles past a row's end but in its last
// group (tiles of 32 x 28 or 64 x 14 cells would cover 32..160-cell boxes 1.3 to 1.4
// times over, the bands 1.13 times).  s_x at x = -1 and x = nx is s_x at nx - 1 and 0
// (s is periodic with phi); a partial last group (nx % VX != 0) evaluates s at
// x = nx from its ghost neighbours, the periodic values.
//
// The plane loop is the row kernel's (fwd_row_kernel): phi around a group stays in
// registers from the sharpening at plane k+1 to the update at plane k+1, every slot
// lies at a compile-time offset (sized for the largest band), unrolled over the four phi
// slots, and four base registers (a row's place and one, two, three pitches on) reach
// every array.  Its expressions in its order: the field is the other kernels' bit for
// bit.
//
// What bounds it: latency (16 warps per SM, one barrier per plane; 54% of the issue slots, the L1
// data pipe at 55%, DRAM at 50% of its rate).  Fewer rows per band, so that no thread has a ring
// group besides its own, took 20% longer; 512 threads, one block per SM, 10%.  64 FP32 boxes with
// edges 32..160 (65 M cells): 143 -> 107 instructions per cell, 341 -> 304 us per step of a run
// (another 64, 58.4 M cells, taller bands: 101.8 and 264 us);
// before, the stores kept ghost cells at both ends of every row, the slots lay at run-time offsets,
// a condition per thread stood around the update, and its operands were loaded after the
// sharpening.  The output goes to the padded copy of the next state and, on the last step of a call
// (final_write), also to the caller's array.
#pragma once

#include "cdi_async.cuh"
#include "cdi_fwd_common.cuh"
#include "cdi_reduce.cuh"
#include "cdi_row.cuh"

namespace cdi {

constexpr int VBAND_NT = 256;  // threads of a vector band block (one cell group each)
constexpr int VBAND_CPY = 2;   // 16-byte vectors of a staged region a thread copies per plane

// Slots (elements), whatever the box: 106 kB, two blocks per SM.
template <typename T>
struct VbandGeo {
    static constexpr int VX = 16 / sizeof(T);
    static constexpr int PHI = VBAND_CPY * VBAND_NT * VX;  // rows y0-2 .. y0+hb+1
    static constexpr int UW = 336 * VX, V = 360 * VX;      // u, w rows y0 ..; v rows y0-1 ..
    static constexpr int VO = UW, WO = UW + V, VEL = 2 * UW + V;
    static constexpr int SX = UW, SY = 400 * VX;           // s_x rows y0 ..; s_y rows y0-1 .. y0+hb
    static constexpr int NPHI = 4, NVEL = 3;
    static constexpr int OVEL = NPHI * PHI, OSX = OVEL + NVEL * VEL, OSY = OSX + 2 * SX;
    static constexpr size_t bytes = sizeof(T) * (size_t)(OSY + 2 * SY);
    static_assert(VEL >= PHI, "the prologue's first phi plane borrows a velocity slot");
};

// Padded layout of a box: row pitch in elements (VX = 16 / sizeof(T)).
__host__ __device__ inline int vband_pitch(int nx, int vx) { return (nx + 2 + vx - 1) / vx * vx; }

// Rows per band: as many whole rows as there are thread groups for and as fit in the slots
// with sv vectors per staged row, with one 4-byte copy per thread (2 (hb + 4) + hb of them).
// 0: a row is too wide (then the body does not apply).
__host__ __device__ inline int vband_rows(int nx, int ny, int vx, int sv)
{
    if (nx > 100 * vx) return 0;
    int hb = VBAND_NT / ((nx + vx - 1) / vx);
    const int cap[] = {VBAND_CPY * VBAND_NT / sv - 4, 336 / sv, 360 / sv - 1, 400 / sv - 2, (VBAND_NT - 8) / 3, ny};
    for (int c : cap) hb = c < hb ? c : hb;
    return hb;
}

// Vectors of a staged row: the row and a vector left of it -- or G + 8 for G groups, where that
// costs no rows of the band: eight lanes of a 16-byte access that straddle two rows then hit
// different banks.
__host__ __device__ inline int vband_staged(int nx, int ny, int vx)
{
    const int sv = vband_pitch(nx, vx) / vx + 1, g = (nx + vx - 1) / vx;
    return g % 8 && vband_rows(nx, ny, vx, g + 8) == vband_rows(nx, ny, vx, sv) ? g + 8 : sv;
}

// The arrays of a unit: padded copies, plane stride P ny, pu | pv | pw vstride apart; raw: the
// caller's array, written too (nullable).
template <typename T>
struct VbandIO {
    const T *pin, *pu;
    T *pout, *raw;
    long long vstride;
    int P, PS;      // row pitch, and that of a staged row
};

template <typename T>
__device__ __forceinline__ void vband_unit(const FwdArgs<T> &a, const VbandIO<T> &io, int y0, int hb, int z0, int z1,
                                           Acc<T> &acc, T *const sm)
{
    using C = VbandGeo<T>;
    constexpr int VX = C::VX, NT = VBAND_NT, ES = sizeof(T);
    using VV = V16<T>;

    const int tid = threadIdx.x;
    const int nx = a.nx, ny = a.ny, nz = a.nz, P = io.P, PS = io.PS;
    const long long planeP = (long long)P * ny;        // padded plane
    unsigned *const st = a.red.status;
    (void)st;
    const T c_adv = a.c.c_adv, c_dif = a.c.c_dif, c_shp = a.c.c_shp, c_upd = a.c.c_upd;

    const int G = (nx + VX - 1) / VX;    // groups per row
    const int hbe = min(hb, ny - y0);    // rows of this band
    // This thread owns group j of band row r.  Warps with such threads run the loop with the
    // update, their lanes past the band on its last group (the same values to the same places, no
    // output); the others the loop without it.  (A condition per thread around the update instead
    // copied every carried value at its end: 15 moves per cell.)
    const int own = min(tid, hbe * G - 1);
    const bool act = (tid & ~31) < hbe * G;
    const int r = own / G, j = own - r * G;
    const int x0 = j * VX;
    const int nown = tid < hbe * G ? min(VX, nx - x0) : 0;  // cells of the group inside the row
    // b0 + q PS: the group in row r + q of an array, so phi row r - 2 + q, u, w, s_x row r + q,
    // v, s_y row r - 1 + q
    T *const b0 = sm + r * PS + VX + x0;
    T *const b1 = b0 + PS, *const b2 = b1 + PS, *const b3 = b2 + PS;
    // s_x left of x = 0 is s_x(nx - 1), right of x = nx - 1 (full last group) s_x(0)
    const T *const sL = b0 + (x0 == 0 ? nx - 1 : -1), *const sR = b0 + (x0 + VX == nx ? VX - nx : VX);
    // ring rows (s_y below and above the band): a group each for 2 G threads, those without a
    // group of their own first; rg: its place as b2 is the own group's
    const int l = NT - 1 - tid;
    const bool ring = l < 2 * G;
    T *const rg = sm + (ring ? ((l >= G ? hbe : -1) + 2) * PS + VX + (l >= G ? l - G : l) * VX : PS);

    // this thread's chunks of the staged regions: phi, u and w (same rows), v; ge: its single cell,
    // of phi (2 left of each row) or of u (1 left of each row)
    int gphi[VBAND_CPY], guw[VBAND_CPY], gv[VBAND_CPY], ge = 0;
    unsigned d[VBAND_CPY], de;  // shared byte addresses
    const int nv = P / VX;
#pragma unroll
    for (int i = 0; i < VBAND_CPY; ++i) {
        const int c = tid + i * NT, row = c / nv, col = (c - row * nv) * VX;
        auto at = [&](int yb, int rows) { return row < rows ? CDI_CHK(wrapi(yb + row, ny), ny, st) * P + col : -1; };
        gphi[i] = at(y0 - 2, hbe + 4);
        guw[i] = at(y0, hbe);
        gv[i] = at(y0 - 1, hbe + 1);
        d[i] = smem_addr(sm + (row < hbe + 4 ? row * PS + VX + col : 0));
    }
    const bool ephi = tid < 2 * (hbe + 4), eu = !ephi && tid < 2 * (hbe + 4) + hbe;
    {
        const int row = ephi ? tid >> 1 : eu ? tid - 2 * (hbe + 4) : 0, x = ephi ? -1 - (tid & 1) : -1;
        ge = CDI_CHK(wrapi(y0 + row - (ephi ? 2 : 0), ny), ny, st) * P + wrapi(x, nx);
        de = smem_addr(sm + row * PS + VX + x);
    }
    int zq = wrapi(z0 - 2, nz);  // wrapped index of the next phi plane to stage
    auto next_phi = [&](auto SO) {
        constexpr int so = decltype(SO)::value * ES;
        const T *const src = io.pin + (long long)CDI_CHK(zq, nz, st) * planeP;
#pragma unroll
        for (int i = 0; i < VBAND_CPY; ++i)
            if (gphi[i] >= 0) cp_async_at<16, so>(d[i], src + gphi[i]);
        if (ephi) cp_async_at<ES, so>(de, src + ge);
        zq = zq + 1 == nz ? 0 : zq + 1;
    };
    const T *vsrc = io.pu + (long long)CDI_CHK(z0, nz, st) * planeP;  // u at the next velocity plane to stage
    int vis = 0, vrd = 0;  // velocity slots (element offsets) of that plane, and of plane k
    auto next_vel = [&]() {
        constexpr int so = C::OVEL * ES;
        const unsigned vb = vis * ES;
#pragma unroll
        for (int i = 0; i < VBAND_CPY; ++i) {
            if (guw[i] >= 0) {
                cp_async_at<16, so>(d[i] + vb, vsrc + guw[i]);
                cp_async_at<16, so + C::WO * ES>(d[i] + vb, vsrc + 2 * io.vstride + guw[i]);
            }
            if (gv[i] >= 0) cp_async_at<16, so + C::VO * ES>(d[i] + vb, vsrc + io.vstride + gv[i]);
        }
        if (eu) cp_async_at<ES, so>(de + vb, vsrc + ge);
        vsrc += planeP;
        vis = vis == 2 * C::VEL ? 0 : vis + C::VEL;
    };

    // Sharpening of the cells c, from the y neighbours, the planes below (zn) and above (zp)
    // and the x neighbours L, R.
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

    // Slot of phi plane z: (z - z0) mod 4; of its velocities: (z - z0) mod 3.
    __syncthreads();  // the previous unit's readers are done with every slot
    next_vel();
    T wlo[VX];  // w on the face below plane z0 (own cells)
    VV::ld(wlo, io.pu + 2 * io.vstride + wrapi(z0 - 1, nz) * planeP + (long long)(y0 + r) * P + x0);
    // planes z0-2 (in the velocity slot of plane z0+2, free until then), z0-1 .. z0+2
    constexpr int M2 = C::OVEL + 2 * C::VEL;
    next_phi(IC<M2>{});
    next_phi(IC<3 * C::PHI>{});
    next_phi(IC<0>{});
    next_phi(IC<C::PHI>{});
    next_phi(IC<2 * C::PHI>{});
    cp_async_commit();
    if (z0 + 1 < z1) next_vel();
    cp_async_commit();
    cp_async_wait<1>();
    __syncthreads();

    // Prologue: s_z at plane z0-1 (own), s at plane z0 (own + ring), flux at z0-1/2.
    // Carried: cK, ynK, ypK, LK, RK phi around the group at plane k; cN the group at plane
    // k+1; sxK, szK its s_x, s_z at plane k; Fzm the flux through its lower z faces; rK the
    // ring group at plane k.
    T cK[VX], cN[VX], ynK[VX], ypK[VX], LK, RK, sxK[VX], szK[VX], Fzm[VX], rK[VX];
    if (ring) {
        T c[VX], yn[VX], yp[VX], zn[VX], zp[VX], s0[VX], s1[VX], s2[VX];
        VV::ld(c, rg);
        VV::ld(yn, rg - PS);
        VV::ld(yp, rg + PS);
        VV::ld(zn, rg + 3 * C::PHI);
        VV::ld(zp, rg + C::PHI);
        sharp(c, yn, yp, zn, zp, rg[-1], rg[VX], s0, s1, s2);
        VV::st(rg - PS + C::OSY, s1);
#pragma unroll
        for (int i = 0; i < VX; ++i) rK[i] = c[i];
    }
    if (act) {
        VV::ld(cK, b2);
        VV::ld(ynK, b1);
        VV::ld(ypK, b3);
        VV::ld(cN, b2 + C::PHI);
        LK = b2[-1];
        RK = b2[VX];
        T cm[VX], s1[VX];
        VV::ld(cm, b2 + 3 * C::PHI);
        sharp(cK, ynK, ypK, cm, cN, LK, RK, sxK, s1, szK);
        VV::st(b1 + C::OSY, s1);
        VV::st(b0 + C::OSX, sxK);
        T ym[VX], yq[VX], zm[VX], a0[VX], a1[VX], szm[VX];
        VV::ld(ym, b1 + 3 * C::PHI);
        VV::ld(yq, b3 + 3 * C::PHI);
        VV::ld(zm, b2 + M2);
        sharp(cm, ym, yq, zm, cK, b2[3 * C::PHI - 1], b2[3 * C::PHI + VX], a0, a1, szm);
#pragma unroll
        for (int i = 0; i < VX; ++i) Fzm[i] = flux(c_adv * wlo[i], c_dif, c_shp, cm[i], cK[i], szm[i], szK[i]);
    }
    __syncthreads();  // the slots of planes z0-2 and z0-1 are free
    if (z0 + 3 <= z1 + 1) next_phi(IC<3 * C::PHI>{});
    cp_async_commit();

    // the group at plane k of the output, and of the caller's array
    T *op = io.pout + (long long)z0 * planeP + (long long)(y0 + r) * P + x0;
    T *raw = io.raw ? io.raw + (long long)z0 * nx * ny + (long long)(y0 + r) * nx + x0 : nullptr;
    const bool raw_v = nx % VX == 0 && ((size_t)io.raw & 15) == 0;
    // One plane: S = (k - z0) mod 4; ACT: with the update.
    auto body = [&](auto SC, auto ACT, const int k) {
        constexpr int S = decltype(SC)::value, S1 = (S + 1) & 3, S2 = (S + 2) & 3;
        constexpr int b = S & 1, bn = b ^ 1;
        // phi plane k+2 and the velocities of plane k have landed, and every thread
        // has left iteration k-1
        cp_async_wait<1>();
        asm volatile("bar.sync 0;" ::: "memory");  // (met from both loops)
        if (k + 4 <= z1 + 1) next_phi(IC<S * C::PHI>{});
        if (k + 2 < z1) next_vel();
        cp_async_commit();

        // sharpening at plane k+1: the ring rows, then the own group
        if (ring) {
            const T *const R1 = rg + S1 * C::PHI;
            T c[VX], yn[VX], yp[VX], zp[VX], s0[VX], s1[VX], s2[VX];
            VV::ld(c, R1);
            VV::ld(yn, R1 - PS);
            VV::ld(yp, R1 + PS);
            VV::ld(zp, rg + S2 * C::PHI);
            sharp(c, yn, yp, rK, zp, R1[-1], R1[VX], s0, s1, s2);
            VV::st(rg - PS + C::OSY + bn * C::SY, s1);
#pragma unroll
            for (int i = 0; i < VX; ++i) rK[i] = c[i];
        }
        if constexpr (decltype(ACT)::value) {
            T cP[VX], ynN[VX], ypN[VX], sxN[VX], szN[VX];
            VV::ld(cP, b2 + S2 * C::PHI);
            VV::ld(ynN, b1 + S1 * C::PHI);
            VV::ld(ypN, b3 + S1 * C::PHI);
            const T LN = b2[S1 * C::PHI - 1], RN = b2[S1 * C::PHI + VX];
            // the update's operands too, before the stores below (the compiler would not move a load
            // over them): their latency passes under the sharpening
            T syn[VX], syp[VX], uc[VX], vc[VX], vn[VX], wc[VX];
            VV::ld(syn, b0 + C::OSY + b * C::SY);
            VV::ld(syp, b2 + C::OSY + b * C::SY);
            const T *const v0 = b0 + vrd;
            VV::ld(uc, v0 + C::OVEL);
            VV::ld(vn, v0 + C::OVEL + C::VO);
            VV::ld(vc, b1 + vrd + C::OVEL + C::VO);
            VV::ld(wc, v0 + C::OVEL + C::WO);
            const T sxL = sL[C::OSX + b * C::SX], sxR = sR[C::OSX + b * C::SX], uL = v0[C::OVEL - 1];
            {
                T s1[VX];
                sharp(cN, ynN, ypN, cK, cP, LN, RN, sxN, s1, szN);
                VV::st(b1 + C::OSY + bn * C::SY, s1);
                VV::st(b0 + C::OSX + bn * C::SX, sxN);
            }
            // fluxes and update at plane k (s of plane k: written before the barrier)
            T o[VX];
#pragma unroll
            for (int i = 0; i < VX; ++i) {
                const T xl = i > 0 ? cK[i - 1] : LK, xr = i + 1 < VX ? cK[i + 1] : RK;
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
                o[i] = fma(-c_upd, div, cK[i]);
                Fzm[i] = Fzp;
            }
            acc.template add_group_n<VX>(o, nown, a.c.tol);
            if (nown == VX) {
                VV::st(op, o);
            } else {
#pragma unroll
                for (int i = 0; i < VX - 1; ++i)
                    if (i < nown) op[i] = o[i];
            }
            if (x0 == 0 && nown > 0) {  // the row's continuation
                op[nx] = o[0];
                op[nx + 1] = nx > 1 ? o[1] : o[0];
            }
            if (raw) {  // the caller's array: rows on 16-byte boundaries, or at any element
                if (raw_v) {
                    if (nown > 0) VV::st(raw, o);
                } else {
#pragma unroll
                    for (int i = 0; i < VX; ++i)
                        if (i < nown) raw[i] = o[i];
                }
                raw += (long long)nx * ny;
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
            RK = RN;
        }
        op += planeP;
        vrd = vrd == 2 * C::VEL ? 0 : vrd + C::VEL;
    };
    auto planes = [&](auto ACT) {
        for (int k = z0;;) {
            body(IC<0>{}, ACT, k);
            if (++k == z1) break;
            body(IC<1>{}, ACT, k);
            if (++k == z1) break;
            body(IC<2>{}, ACT, k);
            if (++k == z1) break;
            body(IC<3>{}, ACT, k);
            if (++k == z1) break;
        }
    };
    if (act) planes(IC<1>{});
    else planes(IC<0>{});
    cp_async_wait<0>();
}

}  // namespace cdi
