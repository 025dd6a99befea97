// Steps of a 2D box (nz == 1) held in shared memory: the state stays on chip from the first step
// of a launch to its last, so a step costs its arithmetic and a barrier or two instead of a
// launch, a pass through L2 and a block reduction.
//
// plane_steps advances a band of whole rows [yb, yb + R) of a box by n steps.  MULTI = false: the
// band is the whole box, its periodic neighbours found by wrapping indices.  MULTI = true: the
// box is cut into bands, one per block of a cooperative grid; a band keeps two halo rows on each
// side, evaluates the sharpening of one ring row on each side itself, and exchanges the halo
// rows with its two neighbours once per step.
//
// The exchange has no flags: a value travels as 64-bit words of 32 payload bits and a 32-bit tag
// (the step's number, unique over the launches of a grid), written by the thread that computed
// the value and polled by the thread that needs it, so a halo costs one trip to L2 and back.  Two
// sets of words alternate by step: a band writes a set again only after it has the words its
// neighbour wrote a step later, which that neighbour computed from the set.  Each wait is bounded.
//
// Cells are visited by their linear index in the band, thread t taking cells t, t + NT, ...; the
// arithmetic is flat_unit's expression by expression (terms that are exactly zero left out), so
// the fields are every other kernel's bit for bit.  FACE: the face-product sharpening (the s
// arrays then hold the normals).
#pragma once

#include "cdi_async.cuh"
#include "cdi_fwd_common.cuh"
#include "cdi_reduce.cuh"

namespace cdi {

// Shared values of one band of R rows: phi twice (with halos), s_x, s_y (with ring rows).
__host__ __device__ constexpr long long plane_values(int nx, int R, bool multi)
{
    return (long long)nx * (multi ? 2 * (R + 4) + R + (R + 2) : 4 * R);
}

// Halo words of one value.
template <typename T> struct HaloWord { static constexpr int N = sizeof(T) / 4; };

// Extrema and violation counts only (Acc::add without the sum, which only the last step needs).
__device__ __forceinline__ void add_bounds(Acc<float> &a, float p, float tol)
{
    a.mn = fminf(a.mn, p);
    a.mx = fmaxf(a.mx, p);
    if (p < 0.f || p > 1.f) {
        ++a.ns;
        a.nt += (p < -tol) | (p > 1.f + tol);
    }
}
__device__ __forceinline__ void add_bounds(Acc<double> &a, double p, double tol)
{
    const long long k = okey(p);
    if (Acc<double>::num(k)) {
        a.kmn = min(a.kmn, k);
        a.kmx = max(a.kmx, k);
        if ((k < KEY_NZERO) | (k > KEY_ONE)) a.count(k, tol);
    }
}

struct PlaneHalo {
    unsigned long long *words;  // [2][bands][2 sides][2 rows][nx][HaloWord]
    int bands, band;
    unsigned tag;               // tag of this launch's first exchanged step
    unsigned long long wait_ns;
    unsigned *status;
    unsigned *gave_up;          // tag of the last launch in which a wait gave up
};

__device__ __forceinline__ void halo_put(unsigned long long *w, unsigned tag, float v)
{
    const unsigned long long x = ((unsigned long long)tag << 32) | __float_as_uint(v);
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(w), "l"(x) : "memory");
}
__device__ __forceinline__ void halo_put(unsigned long long *w, unsigned tag, double v)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(v), t = (unsigned long long)tag << 32;
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(w), "l"(t | (b & 0xffffffffull)) : "memory");
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(w + 1), "l"(t | (b >> 32)) : "memory");
}

// Wait for the word with this tag, for at most h.wait_ns (read from the global timer every few
// polls); gives up at once if a wait of this launch has, else records that and status bit 0 (which
// stays set until the host reads it: a later launch waits for its own words all the same).
__device__ __forceinline__ unsigned halo_word(const unsigned long long *w, unsigned tag, const PlaneHalo &h, bool &ok)
{
    unsigned long long v, t0 = 0;
    for (unsigned i = 0;; ++i) {
        asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(w) : "memory");
        if ((unsigned)(v >> 32) == tag || !ok) return (unsigned)v;
        if ((i & 63u) == 63u) {
            const unsigned long long t = global_ns();
            unsigned gu;
            asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(gu) : "l"(h.gave_up) : "memory");
            if (t0 == 0) t0 = t;
            if (t - t0 > h.wait_ns) {
                atomicOr(h.status, 1u);
                atomicExch(h.gave_up, h.tag);
                ok = false;
            } else if (gu == h.tag) {
                ok = false;
            }
        }
    }
}
__device__ __forceinline__ float halo_get(const unsigned long long *w, unsigned tag, const PlaneHalo &h, bool &ok, float)
{
    return __uint_as_float(halo_word(w, tag, h, ok));
}
__device__ __forceinline__ double halo_get(const unsigned long long *w, unsigned tag, const PlaneHalo &h, bool &ok,
                                           double)
{
    const unsigned lo = halo_word(w, tag, h, ok), hi = halo_word(w + 1, tag, h, ok);
    return __longlong_as_double((long long)(((unsigned long long)hi << 32) | lo));
}

// n steps of rows [yb, yb + R) of the box a (phi -> out; prev, nullable: receives the state one
// step before the last; with n == 1, phi itself).  c_adv(s): the advective coefficient of step s.
// run collects the bounds of every step, last the statistics of the last one.
template <typename T, int NT, bool FACE, bool MULTI, typename CA>
__device__ __forceinline__ void plane_steps(const PlaneArgs<T> &a, T *prev, int yb, int R, int n, CA c_adv_of,
                                            const PlaneHalo &h, Acc<T> &run, Acc<T> &last, T *sm)
{
    constexpr int HL = MULTI ? 2 : 0, RL = MULTI ? 1 : 0;  // halo rows of phi, ring rows of s_y
    const int nx = a.nx, ny = a.ny, P = R * nx, FP = (R + 2 * HL) * nx;
    T *cur = sm, *nxt = sm + FP;
    T *const ssx = sm + 2 * FP, *const ssy = ssx + P;      // ssy from row -RL
    const int tid = threadIdx.x;
    const T c_dif = a.c.c_dif, c_shp = a.c.c_shp, c_upd = a.c.c_upd;
    const int dx = NT % nx, dy = NT / nx;                  // a thread's next cell
    const long long own0 = (long long)yb * nx;
    bool ok = true;

    auto advance = [&](int &x, int &y) {
        x += dx;
        y += dy;
        if (x >= nx) {
            x -= nx;
            ++y;
        }
    };
    // neighbours of cell l (column x, row y of the band) as offsets in its array
    auto left = [&](int x) { return x == 0 ? nx - 1 : -1; };
    auto right = [&](int x) { return x == nx - 1 ? 1 - nx : 1; };
    auto down = [&](int y) { return !MULTI && y == 0 ? P - nx : -nx; };
    auto up = [&](int y) { return !MULTI && y == R - 1 ? nx - P : nx; };

    __syncthreads();  // the buffers' previous readers are done
    for (int l = tid, x = tid % nx, y = tid / nx; l < FP; l += NT, advance(x, y))
        cur[l] = __ldcg(a.phi + (long long)wrapi(yb - HL + y, ny) * nx + x);
    __syncthreads();
    if (prev && n == 1)
        for (int l = tid; l < P; l += NT) prev[own0 + l] = cur[HL * nx + l];

    for (int s = 0; s < n; ++s) {
        const T c_adv = c_adv_of(s);
        // sharpening of the own rows and (s_y) the ring rows
        for (int l = tid, x = tid % nx, y = tid / nx; l < (R + 2 * RL) * nx; l += NT, advance(x, y)) {
            const T *const p = cur + (HL - RL) * nx + l;
            const T c = p[0];
            const T g0 = p[right(x)] - p[left(x)];
            const T g1 = p[up(y)] - p[down(y)];
            const T q = fma(g1, g1, fma(g0, g0, NumLim<T>::tiny()));
            const T inv = rsqrt_t(q);
            const T wgt = FACE ? inv : c * (T(1) - c) * inv;
            if (!MULTI || (y >= RL && y < R + RL)) ssx[l - RL * nx] = wgt * g0;
            ssy[l] = wgt * g1;
        }
        __syncthreads();
        const bool fin = s == n - 1;
        T *const gout = fin ? a.out : s == n - 2 ? prev : nullptr;
        for (int l = tid, x = tid % nx, y = tid / nx; l < P; l += NT, advance(x, y)) {
            const T *const p = cur + HL * nx + l, *const sx = ssx + l, *const sy = ssy + RL * nx + l;
            const int L = left(x), Rr = right(x), D = down(y), U = up(y);
            const T pc = p[0], pxm = p[L], pxp = p[Rr], pym = p[D], pyp = p[U];
            const T sxm = sx[L], sxp = sx[Rr], sym = sy[D], syp = sy[U];
            const T *const u = a.u + own0 + l, *const v = a.v + own0 + l;
            const T uc = __ldg(u), um = __ldg(u + L), vc = __ldg(v);
            const T vm = __ldg(yb + y == 0 ? v + (long long)(ny - 1) * nx : v - nx);
            T adv = uc * (pc + pxp);
            adv = fma(-um, pxm + pc, adv);
            adv = fma(vc, pc + pyp, adv);
            adv = fma(-vm, pym + pc, adv);
            const T dif = fma(T(-4), pc, (pxm + pxp) + (pym + pyp));
            T shp;
            if constexpr (FACE) {
                const T nxc = sx[0], nyc = sy[0];
                const T fxp = T(0.5) * (pc + pxp), fxm = T(0.5) * (pxm + pc);
                const T fyp = T(0.5) * (pc + pyp), fym = T(0.5) * (pym + pc);
                shp = (fxp * (T(1) - fxp) * (nxc + sxp) - fxm * (T(1) - fxm) * (sxm + nxc)) +
                      (fyp * (T(1) - fyp) * (nyc + syp) - fym * (T(1) - fym) * (sym + nyc));
            } else {
                shp = (sxp - sxm) + (syp - sym);
            }
            const T div = fma(c_adv, adv, fma(-c_dif, dif, c_shp * shp));  // z faces: equal
            const T o = fma(-c_upd, div, pc);
            nxt[HL * nx + l] = o;
            add_bounds(run, o, a.c.tol);
            if (gout) gout[own0 + l] = o;
            if (fin) last.add(o, a.c.tol);
            if constexpr (MULTI) {
                if (!fin) {  // rows 0, 1 for the band below, the last two for the band above
                    unsigned long long *const w =
                        h.words + ((size_t)((s & 1) * h.bands + h.band) * 4 * nx + x) * HaloWord<T>::N;
                    if (y < 2) halo_put(w + (size_t)y * nx * HaloWord<T>::N, h.tag + s, o);
                    if (y >= R - 2) halo_put(w + (size_t)(2 + y - (R - 2)) * nx * HaloWord<T>::N, h.tag + s, o);
                }
            }
        }
        if constexpr (MULTI) {
            if (!fin) {  // rows -2, -1 from the band below (its last two), R, R + 1 from the band above
                for (int l = tid, x = tid % nx, y = tid / nx; l < 4 * nx; l += NT, advance(x, y)) {
                    const int b = y < 2 ? (h.band == 0 ? h.bands - 1 : h.band - 1) : (h.band + 1 == h.bands ? 0 : h.band + 1);
                    const int row = y < 2 ? 2 + y : y - 2;
                    const unsigned long long *const w =
                        h.words + ((size_t)((s & 1) * h.bands + b) * 4 * nx + (size_t)row * nx + x) * HaloWord<T>::N;
                    nxt[(y < 2 ? y : R + y) * nx + x] = halo_get(w, h.tag + s, h, ok, T(0));
                }
            }
        }
        __syncthreads();
        T *const t = cur;
        cur = nxt;
        nxt = t;
    }
}

}  // namespace cdi
