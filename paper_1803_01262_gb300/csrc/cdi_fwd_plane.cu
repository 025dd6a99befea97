// Runs of a 2D grid (nz == 1) as one launch: bands of whole rows, one per block of a cooperative
// grid, stepped in shared memory with halo exchange between neighbouring bands (cdi_plane.cuh).
//
// With a launch per step a small plane's step was launch and ramp: 5.8-6.5 us in FP32 from 64^2 to
// 256^2 (8.2 on the one-cell-per-thread tiles), 21 us in FP64.  Held on chip, a run of 32 steps
// takes 1.5 us per step at 128^2, 1.7 at 256^2 (an exchange between neighbours, about 1 us, and
// two block barriers) and 8.7 at 1024^2 (20.5 before); FP64 5.3 us at 128^2 and 26 at 512^2 (60
// before), where the FP64 pipe of all SMs bounds it.
#include "cdi_internal.cuh"
#include "cdi_plane.cuh"

namespace cdi {

template <typename T>
struct PlaneCoefs {
    T c_adv[kPlaneSteps];
};

template <typename T, int NT, bool MULTI>
__global__ void __launch_bounds__(NT)
fwd_plane_kernel(const PlaneArgs<T> a, const RedScratch red, T *prev, const int n, const __grid_constant__ PlaneCoefs<T> cs,
                 unsigned long long *words, unsigned *tag, const unsigned long long wait_ns)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int is_last;
    const int tid = threadIdx.x, b = blockIdx.x, B = gridDim.x;
    const int yb = (int)((long long)b * a.ny / B), R = (int)((long long)(b + 1) * a.ny / B) - yb;
    const unsigned base = *tag;  // (moved on by the last block of the launch, below)
    Acc<T> run, last;
    run.init();
    last.init();
    const PlaneHalo h = {words, B, b, base, wait_ns, red.status, tag + 1};
    plane_steps<T, NT, false, MULTI>(a, prev, yb, R, n, [&](int s) { return cs.c_adv[s]; }, h, run, last,
                                     reinterpret_cast<T *>(smem_raw));
    // the last step's statistics into the record, every step's bounds into the run's
    const Partial pl = block_partial(last), pr = block_partial(run);
    if (tid == 0) {
        red.partials[b] = pl;
        red.partials[B + b] = pr;
        __threadfence();
        is_last = atomicAdd(red.counter, 1u) == (unsigned)(B - 1);
    }
    __syncthreads();
    if (!is_last) return;
    __threadfence();
    constexpr bool F32 = sizeof(T) == 4;
    StatsRec *const r = red.rec;
    StatsRec o;
    if (tid == 0) {
        o.mn_run = __ldcg(&r->mn_run);
        o.mx_run = __ldcg(&r->mx_run);
        o.ns_run = __ldcg(&r->ns_run);
        o.nt_run = __ldcg(&r->nt_run);
        o.steps_run = __ldcg(&r->steps_run);
    }
    const Partial q = combine_partials<F32>(red.partials, B), qr = combine_partials<F32>(red.partials + B, B);
    if (tid == 0) {
        r->sum = q.sum;
        r->mn = q.mn;
        r->mx = q.mx;
        r->ns = q.ns;
        r->nt = q.nt;
        r->mass = red.dV * q.sum;
        r->mn_run = fmin(o.mn_run, qr.mn);
        r->mx_run = fmax(o.mx_run, qr.mx);
        r->ns_run = o.ns_run + qr.ns;
        r->nt_run = o.nt_run + qr.nt;
        r->steps_run = o.steps_run + n;
        *red.counter = 0u;
        *tag = base + (unsigned)n;
    }
}

// A wait for words that no block writes: it must run out after wait_ns.  The tag moves on, as after a run.
__global__ void halo_probe_kernel(const unsigned long long *words, unsigned *tag, unsigned *status,
                                  const unsigned long long wait_ns)
{
    const PlaneHalo h = {nullptr, 1, 0, *tag, wait_ns, status, tag + 1};
    bool ok = true;
    (void)halo_word(words, h.tag + 0x40000000u, h, ok);
    __syncthreads();
    if (threadIdx.x == 0) *tag = h.tag + 1u;
}

cudaError_t launch_halo_probe(const unsigned long long *words, unsigned *tag, unsigned *status,
                              unsigned long long wait_ns, cudaStream_t s)
{
    halo_probe_kernel<<<1, 32, 0, s>>>(words, tag, status, wait_ns);
    return cudaGetLastError();
}

// 512 threads per band (256: 1.75, 1024: 1.77 against 1.60 us per step at 128^2 FP32).
constexpr int kPlaneNT = 512;

template <typename T>
static cudaError_t plane_smem(size_t *lim)
{
    int dev = 0, optin = 0;
    cudaFuncAttributes fa;
    cudaError_t e;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess ||
        (e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev)) != cudaSuccess ||
        (e = cudaFuncGetAttributes(&fa, fwd_plane_kernel<T, kPlaneNT, true>)) != cudaSuccess)
        return e;
    *lim = (size_t)optin - fa.sharedSizeBytes;
    return cudaSuccess;
}

template <typename T>
cudaError_t plane_bands(int nx, int ny, int sms, int *bands, size_t *smem)
{
    *bands = 0;
    size_t lim = 0;
    cudaError_t e = plane_smem<T>(&lim);
    if (e != cudaSuccess) return e;
    // Bands of about 256 cells and at least the two rows a neighbour's halo takes: an exchange
    // costs ~1 us whatever the band, so a step wants few cells per block until the SMs run out
    // (128^2 FP64: 5.3 us per step with 256 cells, 7.6 with 512, 12.2 with 1024; FP32 1.49, 1.60,
    // 1.80).
    int rows = (256 + nx - 1) / nx;
    if (rows < 2) rows = 2;
    int B = ny / rows;
    if (B > sms) B = sms;
    if (B < 2) B = 1;
    const int R = (ny + B - 1) / B;
    const size_t need = sizeof(T) * (size_t)plane_values(nx, R, B > 1);
    if (need > lim) return cudaSuccess;
    *bands = B;
    *smem = need;
    e = cudaFuncSetAttribute(fwd_plane_kernel<T, kPlaneNT, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)lim);
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(fwd_plane_kernel<T, kPlaneNT, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)lim);
}

template <typename T>
size_t plane_word_bytes(int nx, int bands)
{
    return (size_t)2 * bands * 4 * nx * HaloWord<T>::N * sizeof(unsigned long long);
}

template <typename T>
cudaError_t launch_fwd_plane(const PlaneArgs<T> &a, const RedScratch &red, T *prev, int n, const T *c_adv, int bands,
                             size_t smem, unsigned long long *words, unsigned *tag, cudaStream_t s)
{
    PlaneCoefs<T> cs;
    for (int i = 0; i < n; ++i) cs.c_adv[i] = c_adv[i];
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)bands);
    cfg.blockDim = dim3(kPlaneNT);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeCooperative;  // the bands wait on one another
    at[0].val.cooperative = 1;
    cfg.attrs = at;
    cfg.numAttrs = bands > 1 ? 1 : 0;
    const unsigned long long wait_ns = 1000000000ull;  // a step takes microseconds
    if (bands > 1)
        return cudaLaunchKernelEx(&cfg, fwd_plane_kernel<T, kPlaneNT, true>, a, red, prev, n, cs, words, tag, wait_ns);
    return cudaLaunchKernelEx(&cfg, fwd_plane_kernel<T, kPlaneNT, false>, a, red, prev, n, cs, words, tag, wait_ns);
}

template cudaError_t plane_bands<float>(int, int, int, int *, size_t *);
template cudaError_t plane_bands<double>(int, int, int, int *, size_t *);
template size_t plane_word_bytes<float>(int, int);
template size_t plane_word_bytes<double>(int, int);
template cudaError_t launch_fwd_plane<float>(const PlaneArgs<float> &, const RedScratch &, float *, int, const float *,
                                             int, size_t, unsigned long long *, unsigned *, cudaStream_t);
template cudaError_t launch_fwd_plane<double>(const PlaneArgs<double> &, const RedScratch &, double *, int,
                                              const double *, int, size_t, unsigned long long *, unsigned *,
                                              cudaStream_t);

}  // namespace cdi
