// Tile geometry and staging shared by the row kernels (forward, adjoint): tiles of W x TY cells
// (W = 16 vectors of 16 bytes), own warp w holding rows 2w and 2w + 1, one vector per thread,
// and a last warp for the one-cell ring; planes staged by cp.async into rings of four slots
// whose offsets are compile-time constants, every array with one row pitch.
#pragma once

#include <type_traits>

#include "cdi_async.cuh"
#include "cdi_fwd_common.cuh"

namespace cdi {

template <int V>
using IC = std::integral_constant<int, V>;

template <typename T, int TY>
struct RowGeo {
    static constexpr int VX = 16 / sizeof(T), TX = 16;
    static constexpr int W = TX * VX, H = TY;
    static constexpr int NOWN = TX * TY;
    static constexpr int NT = NOWN + 32;      // + the ring warp
    static constexpr int NJ = W / 32;         // a lane's columns of a row
    static constexpr int PP = W + 2 * VX;     // row pitch of every staged array: x0-VX .. x0+W+VX-1
    static constexpr int NS = 4;              // ring slots
    static constexpr int PHI = (H + 4) * PP;  // a halo-2 plane (phi, lam'): rows y0-2 .. y0+H+1
    static constexpr int VO = H * PP;         // velocities: u rows y0 .. at 0; v rows y0-1 ..; w rows y0 ..
    static constexpr int WO = VO + (H + 1) * PP;
    static constexpr int VEL = WO + H * PP;
    static constexpr int SXS = H * PP;        // an x-exchanged array, columns -1 .. W
    static constexpr int SYS = (H + 2) * PP;  // a y-exchanged array, rows -1 .. H
    static_assert(TY % 2 == 0 && TY <= 14, "two rows per own warp, at most 60 single halo cells");
};

// Copies of one work unit: in-plane offsets planned once, then a plane's copies are a base
// pointer and immediates.  Own threads, AL: g[0] the own vector; else (A elements per copy:
// 1, or 2 where rows start on pairs) g[r NJ + j] column A (lane + 32 j) of row r0 + r.  Ring warp, AL: g[0..2] / d[0..2] vectors of a halo-2 plane (rows -1
// and H with their x halos, rows -2 and H+1, the x halos of rows 0..H-1), g[3] / d[3] the x halo
// of u (lanes < H) and v row -1 (16 lanes).  Else g[r NJ + j] the rows -2, -1, H, H+1, gv[j] v
// row -1, gh[0..1] / d[0..1] single cells (columns -1 and W of rows -1 and H; columns -2, -1, W,
// W+1 of rows 0..H-1; A = 2: pairs left and right of rows -1 .. H), gh[2] / d[2] u column -1.
template <typename T, int TY, int A>
struct RowStage {
    using G = RowGeo<T, TY>;
    static constexpr bool AL = A == G::VX, PR = !AL && A == 2;
    static constexpr int EB = A * sizeof(T);  // bytes of a copy by elements
    static constexpr int VX = G::VX, W = G::W, H = G::H, PP = G::PP, NJ = G::W / 32 / (AL ? 1 : A), ES = sizeof(T);
    static constexpr int NG = AL ? 4 : 4 * NJ;
    int g[NG], gh[3], gv[NJ];
    unsigned d[4];     // shared byte addresses of the ring warp's single places
    unsigned cb;       // base shared address: own threads, AL: the own vector's place (below);
                       // else column `lane` of the warp's first row (ring warp: of row 0)
    bool is_own, hx2;  // hx2: ring warp, AL: its third vector exists
    int lane;
    int pf;  // AL = false, lanes < 6 of an own warp: the cell `ahead` asks for

    // sm: the block's shared memory; row r of a halo-2 plane lands at (r + 2) PP, of u and w at
    // r PP, of v at (r + 1) PP of its region, column c at VX + c
    __device__ __forceinline__ RowStage(T *sm, int tid, int ty, int tx)
    {
        is_own = tid < G::NOWN;
        lane = tid & 31;
        cb = smem_addr(AL ? sm + (ty + 1) * PP + VX + tx * VX : sm + (is_own ? (ty & ~1) * PP : 0) + VX + lane * A);
    }

    __device__ __forceinline__ void plan(T *sm, int x0, int y0, int ty, int tx, int nx, int ny, long long plane,
                                         unsigned *st)
    {
        (void)st;
        hx2 = false;
        pf = 0;
        if (!AL && is_own && lane < 6)
            pf = (int)CDI_CHK(wrapi(y0 + (ty & ~1) + lane / 3, ny) * nx + min(x0 + (lane % 3) * 32, nx - 1), plane, st);
        const int r0 = ty & ~1;
        auto at = [&](int y, int x, int len) {  // wrapped in-plane offset (len elements long)
            return (int)CDI_CHK(wrapi(y, ny) * nx + wrapi(x, nx), plane - len + 1, st);
        };
        if (is_own) {
            if constexpr (AL) {
                g[0] = at(y0 + ty, x0 + tx * VX, VX);
            } else {
#pragma unroll
                for (int r = 0; r < 2; ++r)
#pragma unroll
                    for (int j = 0; j < NJ; ++j) g[r * NJ + j] = at(y0 + r0 + r, x0 + (lane + 32 * j) * A, A);
            }
        } else if constexpr (AL) {
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                int e = lane + 32 * i, row, col;  // col: vector column -1 .. 16
                if (e < 36) {
                    row = e < 18 ? -1 : H;
                    col = e % 18 - 1;
                } else if (e < 68) {
                    e -= 36;
                    row = e < 16 ? -2 : H + 1;
                    col = e & 15;
                } else {
                    e -= 68;  // (rows past H - 1, for TY < 14: a row the tile stages anyway, not copied)
                    row = e >> 1;
                    col = (e & 1) ? 16 : -1;
                }
                g[i] = at(y0 + row, x0 + col * VX, VX);
                hx2 = lane + 32 * i < 68 || row < H;
                d[i] = smem_addr(sm + (hx2 ? (row + 2) * PP + VX + col * VX : 0));
            }
            const bool isu = lane < H;
            g[3] = isu ? at(y0 + lane, x0 - VX, VX) : at(y0 - 1, x0 + ((lane - H) & 15) * VX, VX);
            d[3] = smem_addr(sm + (isu ? lane * PP : G::VO + VX + ((lane - H) & 15) * VX));
        } else {
#pragma unroll
            for (int r = 0; r < 4; ++r)
#pragma unroll
                for (int j = 0; j < NJ; ++j)
                    g[r * NJ + j] = at(y0 + (r < 2 ? r - 2 : H + r - 2), x0 + (lane + 32 * j) * A, A);
#pragma unroll
            for (int j = 0; j < NJ; ++j) gv[j] = at(y0 - 1, x0 + (lane + 32 * j) * A, A);
            if constexpr (PR) {  // pairs left and right of rows -1 .. H
                const int row = lane < 2 * H + 4 ? lane / 2 - 1 : 0, col = lane & 1 ? W : -2;
                gh[0] = at(y0 + row, x0 + col, 2);
                d[0] = smem_addr(sm + (row + 2) * PP + VX + col);
            } else {
#pragma unroll
            for (int i = 0; i < 2; ++i) {  // 4 H + 4 <= 64 cells
                const int e = lane + 32 * i - 4;
                const int row = e < 0 ? (e & 2 ? H : -1) : e >> 2, q = e & 3;
                const int col = e < 0 ? (e & 1 ? W : -1) : q < 2 ? q - 2 : W + q - 2;
                gh[i] = at(y0 + row, x0 + col, 1);
                d[i] = smem_addr(sm + (e < 4 * H ? (row + 2) * PP + VX + col : 0));
            }
            }
            gh[2] = at(y0 + (lane < H ? lane : 0), x0 - 1, 1);
            d[2] = smem_addr(sm + (lane < H ? lane : 0) * PP + VX - 1);
        }
    }

    // AL = false: ask for the own warp's two rows of a plane (src its first element) in L2, a
    // line at a time.  The element copies pass through L1, whose lines (what shared memory leaves
    // of it) bound the bytes in flight; with the rows in L2 a copy holds its line for an L2, not a
    // memory, latency.  For the adjoint without velocity gradients, whose rings leave L1 the least:
    // 255^3 FP32 109 -> 106 us.  (The others gained nothing; cp.async.bulk.prefetch, one per row,
    // took twice as long.)
    __device__ __forceinline__ void ahead(const T *src) const
    {
        if constexpr (!AL) {
            if (is_own && lane < 6) asm volatile("prefetch.global.L2 [%0];" ::"l"(src + pf));
        }
    }

    // A halo-2 plane (src its first element) into the slot at element offset SO.
    template <int SO>
    __device__ __forceinline__ void halo2(const T *src) const
    {
        constexpr int so = SO * ES;
        if (is_own) {
            if constexpr (AL) {
                cp_async_at<16, so + PP * ES>(cb, src + g[0]);
            } else {
                cp_async_at<EB, so + 2 * PP * ES>(cb, src + g[0]);
                cp_async_at<EB, so + 3 * PP * ES>(cb, src + g[NJ]);
                if constexpr (NJ == 2) {
                    cp_async_at<EB, so + (2 * PP + 32) * ES>(cb, src + g[1]);
                    cp_async_at<EB, so + (3 * PP + 32) * ES>(cb, src + g[NJ + 1]);
                }
            }
        } else if constexpr (AL) {
            cp_async_at<16, so>(d[0], src + g[0]);
            cp_async_at<16, so>(d[1], src + g[1]);
            if (TY == 14 || hx2) cp_async_at<16, so>(d[2], src + g[2]);
        } else {
            cp_async_at<EB, so>(cb, src + g[0]);
            cp_async_at<EB, so + PP * ES>(cb, src + g[NJ]);
            cp_async_at<EB, so + (H + 2) * PP * ES>(cb, src + g[2 * NJ]);
            cp_async_at<EB, so + (H + 3) * PP * ES>(cb, src + g[3 * NJ]);
            if constexpr (NJ == 2) {
                cp_async_at<EB, so + 32 * ES>(cb, src + g[1]);
                cp_async_at<EB, so + (PP + 32) * ES>(cb, src + g[NJ + 1]);
                cp_async_at<EB, so + ((H + 2) * PP + 32) * ES>(cb, src + g[2 * NJ + 1]);
                cp_async_at<EB, so + ((H + 3) * PP + 32) * ES>(cb, src + g[3 * NJ + 1]);
            }
            if (lane < (PR ? 2 * H + 4 : 4 * H + 4)) cp_async_at<EB, so>(d[0], src + gh[0]);
            if constexpr (!PR) {
                if (lane + 32 < 4 * H + 4) cp_async_at<EB, so>(d[1], src + gh[1]);
            }
        }
    }

    // Velocity planes (u, v, w at the plane's first element) into the slot at element offset SO.
    template <int SO>
    __device__ __forceinline__ void vel(const T *pu, const T *pv, const T *pw) const
    {
        constexpr int so = SO * ES;
        if (is_own) {
            if constexpr (AL) {
                cp_async_at<16, so - PP * ES>(cb, pu + g[0]);
                cp_async_at<16, so + G::VO * ES>(cb, pv + g[0]);
                cp_async_at<16, so + (G::WO - PP) * ES>(cb, pw + g[0]);
            } else {
                cp_async_at<EB, so>(cb, pu + g[0]);
                cp_async_at<EB, so + PP * ES>(cb, pu + g[NJ]);
                cp_async_at<EB, so + (G::VO + PP) * ES>(cb, pv + g[0]);
                cp_async_at<EB, so + (G::VO + 2 * PP) * ES>(cb, pv + g[NJ]);
                cp_async_at<EB, so + G::WO * ES>(cb, pw + g[0]);
                cp_async_at<EB, so + (G::WO + PP) * ES>(cb, pw + g[NJ]);
                if constexpr (NJ == 2) {
                    cp_async_at<EB, so + 32 * ES>(cb, pu + g[1]);
                    cp_async_at<EB, so + (PP + 32) * ES>(cb, pu + g[NJ + 1]);
                    cp_async_at<EB, so + (G::VO + PP + 32) * ES>(cb, pv + g[1]);
                    cp_async_at<EB, so + (G::VO + 2 * PP + 32) * ES>(cb, pv + g[NJ + 1]);
                    cp_async_at<EB, so + (G::WO + 32) * ES>(cb, pw + g[1]);
                    cp_async_at<EB, so + (G::WO + PP + 32) * ES>(cb, pw + g[NJ + 1]);
                }
            }
        } else if constexpr (AL) {
            if (lane < H + 16) cp_async_at<16, so>(d[3], (lane < H ? pu : pv) + g[3]);
        } else {
            cp_async_at<EB, so + G::VO * ES>(cb, pv + gv[0]);
            if constexpr (NJ == 2) cp_async_at<EB, so + (G::VO + 32) * ES>(cb, pv + gv[1]);
            if (lane < H) cp_async_at<ES, so>(d[2], pu + gh[2]);
        }
    }

    // An own thread's cells of a plane of another array (src its first element) to the W-pitched
    // place at base + SO elements (base: own_base), read back by the same warp.
    __device__ __forceinline__ unsigned own_base(T *sm, int ty, int tx) const
    {
        return smem_addr(sm + (AL ? ty * W + tx * VX : (ty & ~1) * W + lane * A));
    }
    template <int SO>
    __device__ __forceinline__ void own(unsigned base, const T *src) const
    {
        constexpr int so = SO * ES;
        if constexpr (AL) {
            cp_async_at<16, so>(base, src + g[0]);
        } else {
            cp_async_at<EB, so>(base, src + g[0]);
            cp_async_at<EB, so + W * ES>(base, src + g[NJ]);
            if constexpr (NJ == 2) {
                cp_async_at<EB, so + 32 * ES>(base, src + g[1]);
                cp_async_at<EB, so + (W + 32) * ES>(base, src + g[NJ + 1]);
            }
        }
    }
};

// The first n of N cells, A at a time (A = 2: to an address on a pair).
template <int A, int N, typename T>
__device__ __forceinline__ void store_cells(T *p, const T *o, int n)
{
#pragma unroll
    for (int i = 0; i < N; i += A) {
        if (i >= n) continue;
        if constexpr (A == 2 && sizeof(T) == 4) *reinterpret_cast<float2 *>(p + i) = make_float2(o[i], o[i + 1]);
        else p[i] = o[i];
    }
}

}  // namespace cdi
