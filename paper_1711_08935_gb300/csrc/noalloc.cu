// Projection onto one atom's orbitals without any GPU memory allocation.
//
// Some callers cannot allocate device memory at all: code that runs while another component owns
// the whole device memory pool, real-time loops where an allocation (and the device-wide
// synchronisation cudaMalloc/cudaFree may imply) is not allowed, or plug-in code that only receives
// pointers from its host application.  This entry point takes every input and the output as caller
// pointers and keeps its scratch (per-tile partial sums) in a fixed array that is part of the
// library's device image, so nothing is allocated when it runs.
#include <mutex>

#include "dftu_internal.cuh"

namespace {

constexpr int NA_TILE = 512;                          // sphere points per CTA
constexpr int64_t NA_SCRATCH_ELEMS = 524288;          // complex FP64 partial sums: 8 MiB
constexpr int NA_CTA = 128;                           // four warps, each one band of the CTA's chunk
constexpr int NA_MAXDEV = 64;

// Scratch shared by every call on a device; it keeps the previous call's contents.  Every slot a
// call reads is written by the same call first, so nothing needs clearing.
static __device__ __align__(256) double2 g_na_scratch[NA_SCRATCH_ELEMS];

std::mutex g_na_mutex;
double2* g_na_ptr[NA_MAXDEV] = {nullptr};

// One step of the warp's sum of N values per lane: lanes whose bit OFF is clear keep the first half of the
// values, the others the second half, each adding its partner's; the adds of the five steps are N/2 + N/4 + ...
// instead of 5 N, in the order of a plain butterfly.
template <int N, int OFF>
__device__ __forceinline__ void fold(double (&v)[2 * dftu::MAXM], int lane) {
    constexpr int H = (N + 1) / 2;
    const bool up = (lane & OFF) != 0;
#pragma unroll
    for (int i = 0; i < H; ++i) {
        const double lo = v[i], hi = (i + H < N) ? v[i + H] : 0.0;
        const double keep = up ? hi : lo, give = up ? lo : hi;
        v[i] = keep + __shfl_xor_sync(0xffffffffu, give, OFF);
    }
    if constexpr (OFF > 1) fold<H, OFF / 2>(v, lane);
}

// Index of the value that lane ends up with (-1: none).
template <int N, int OFF>
__device__ __forceinline__ int fold_index(int lane) {
    constexpr int H = (N + 1) / 2;
    const bool up = (lane & OFF) != 0;
    int i = 0;
    if constexpr (OFF > 1) i = fold_index<H, OFF / 2>(lane);
    if (i < 0) return -1;
    const int j = up ? i + H : i;
    return j < (up ? N : H) ? j : -1;
}

// partial[tile][band][m] = dV sum_{j in tile} phi[j][m] phase[j] psi[band][idx[j]]   (FP64).
// A grid index outside [0, ld) is never read: the tile then writes NaN partial sums for every band,
// so the projections of the call come out NaN.
// One CTA per (tile, four bands): bound by the FP64 pipe (4 + 2M fused multiply-adds per point and band), so
// the bands are spread over as many CTAs as there are; M is a template argument, which keeps the sums in
// registers.  24405 points, 128 bands, M = 5, complex128: 443 us with all bands of a tile in one CTA and M at
// run time, 91 us now (87 by the fused multiply-adds alone at the measured 0.50 T/s).
template <typename T, int M>
__global__ void __launch_bounds__(NA_CTA) k_na_tiles(const T* __restrict__ psi, int nbands, int64_t ld,
                                                     const int* __restrict__ idx, const double2* __restrict__ phase,
                                                     const double* __restrict__ phi, int npts, double dV,
                                                     double2* __restrict__ part) {
    __shared__ int s_idx[NA_TILE];
    __shared__ double2 s_ph[NA_TILE];
    __shared__ double s_phi[NA_TILE * M];
    __shared__ int s_bad;
    const int ntiles = (npts + NA_TILE - 1) / NA_TILE;   // a flat grid: neither tiles nor bands fit the y axis at the scratch's limit
    const int tile = blockIdx.x % ntiles;
    const int p0 = tile * NA_TILE;
    const int np = min(NA_TILE, npts - p0);
    if (threadIdx.x == 0) s_bad = 0;
    __syncthreads();
    for (int i = threadIdx.x; i < np; i += NA_CTA) {
        const int g = idx[p0 + i];
        const bool ok = g >= 0 && (int64_t)g < ld;
        if (!ok) s_bad = 1;
        s_idx[i] = ok ? g : 0;
        s_ph[i] = phase ? phase[p0 + i] : make_double2(1.0, 0.0);
    }
    for (int e = threadIdx.x; e < np * M; e += NA_CTA) s_phi[e] = phi[(int64_t)p0 * M + e];
    __syncthreads();
    const bool bad = s_bad != 0;
    const int lane = threadIdx.x & 31;
    const int band = blockIdx.x / ntiles * (NA_CTA / 32) + (threadIdx.x >> 5);
    if (band >= nbands) return;
    const T* row = psi + (int64_t)band * ld;
    double v[2 * dftu::MAXM];   // re_0, im_0, re_1, ...
#pragma unroll
    for (int m = 0; m < 2 * M; ++m) v[m] = 0.0;
#pragma unroll 4
    for (int i = lane; i < np; i += 32) {
        const T x = row[s_idx[i]];
        const double xr = (double)x.x, xi = (double)x.y;
        const double2 ph = s_ph[i];
        const double yr = ph.x * xr - ph.y * xi, yi = ph.x * xi + ph.y * xr;
#pragma unroll
        for (int m = 0; m < M; ++m) {
            const double f = s_phi[i * M + m];
            v[2 * m] = fma(f, yr, v[2 * m]);
            v[2 * m + 1] = fma(f, yi, v[2 * m + 1]);
        }
    }
    fold<2 * M, 16>(v, lane);
    const int k = fold_index<2 * M, 16>(lane);
    if (k >= 0) {
        const double nan = __longlong_as_double(0x7FF8000000000000LL);
        reinterpret_cast<double*>(part)[(((int64_t)tile * nbands + band) * M) * 2 + k] = bad ? nan : dV * v[0];
    }
}

// p[band][m] = sum over tiles in order of the partial sums, one thread per real number; eight loads in flight.
__global__ void k_na_reduce(const double* __restrict__ part, int ntiles, int n, double* __restrict__ p) {
    const int g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= n) return;
    double s = 0.0;
    int t = 0;
    for (; t + 8 <= ntiles; t += 8) {
        double x[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) x[q] = part[(int64_t)(t + q) * n + g];
#pragma unroll
        for (int q = 0; q < 8; ++q) s += x[q];
    }
    for (; t < ntiles; ++t) s += part[(int64_t)t * n + g];
    p[g] = s;
}

template <typename T>
const void* tiles_kernel(int M) {
    switch (M) {
        case 1: return reinterpret_cast<const void*>(&k_na_tiles<T, 1>);
        case 2: return reinterpret_cast<const void*>(&k_na_tiles<T, 2>);
        case 3: return reinterpret_cast<const void*>(&k_na_tiles<T, 3>);
        case 4: return reinterpret_cast<const void*>(&k_na_tiles<T, 4>);
        case 5: return reinterpret_cast<const void*>(&k_na_tiles<T, 5>);
        case 6: return reinterpret_cast<const void*>(&k_na_tiles<T, 6>);
        default: return reinterpret_cast<const void*>(&k_na_tiles<T, 7>);
    }
}

// Device address of the scratch array on the current device, looked up once per device.
double2* scratch_for_current_device(int& dev) {
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= NA_MAXDEV) return nullptr;
    std::lock_guard<std::mutex> lock(g_na_mutex);
    if (!g_na_ptr[dev]) {
        void* ptr = nullptr;
        if (cudaGetSymbolAddress(&ptr, g_na_scratch) != cudaSuccess) return nullptr;
        g_na_ptr[dev] = static_cast<double2*>(ptr);
    }
    return g_na_ptr[dev];
}

}  // namespace

extern "C" dftu_status dftu_project_sphere_noalloc(const void* psi, dftu_prec prec, int nbands, int64_t ld_band,
                                                   const int32_t* idx, const double* phase, const double* phi, int npts,
                                                   int M, double dV, double* p_out, dftu_stream stream) {
    if (!psi || !idx || !phi || !p_out || nbands < 1 || npts < 1 || M < 1 || M > dftu::MAXM || !(dV > 0.0) || ld_band < 1 ||
        (prec != DFTU_C128 && prec != DFTU_C64))
        return DFTU_ERR_INVALID_ARG;
    const int ntiles = (npts + NA_TILE - 1) / NA_TILE;
    if ((int64_t)ntiles * nbands * M > NA_SCRATCH_ELEMS) return DFTU_ERR_INVALID_ARG;   // beyond the fixed scratch
    int dev = -1;
    double2* part = scratch_for_current_device(dev);
    if (!part) return DFTU_ERR_CUDA;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    // every operand must be memory this GPU can address (a pageable host array would fault the kernel)
    if (!dftu::gpu_addressable(dev, psi, st) || !dftu::gpu_addressable(dev, idx, st) || !dftu::gpu_addressable(dev, phi, st) ||
        !dftu::gpu_addressable(dev, p_out, st) || (phase && !dftu::gpu_addressable(dev, phase, st)))
        return DFTU_ERR_INVALID_ARG;
    // Launch errors are taken from the launch calls themselves, so an unrelated error the caller left
    // pending is neither reported as ours nor cleared.
    const double2* ph = reinterpret_cast<const double2*>(phase);
    int nt = ntiles;
    void* tile_args[] = {(void*)&psi, (void*)&nbands, (void*)&ld_band, (void*)&idx, (void*)&ph,
                         (void*)&phi, (void*)&npts, (void*)&dV, (void*)&part};
    const void* fn = (prec == DFTU_C128) ? tiles_kernel<double2>(M) : tiles_kernel<float2>(M);
    const int per = NA_CTA / 32;
    const unsigned blocks = (unsigned)ntiles * (unsigned)((nbands + per - 1) / per);   // at most the scratch's size
    cudaError_t e = cudaLaunchKernel(fn, dim3(blocks), dim3(NA_CTA), tile_args, 0, st);
    if (e == cudaSuccess) {
        int n = 2 * nbands * M;
        void* red_args[] = {(void*)&part, (void*)&nt, (void*)&n, (void*)&p_out};
        e = cudaLaunchKernel(reinterpret_cast<const void*>(&k_na_reduce), dim3((n + 127) / 128), dim3(128), red_args, 0, st);
    }
    if (e != cudaSuccess) {
        cudaGetLastError();   // the failed launch is reported here, not left for the caller's next check
        return DFTU_ERR_CUDA;
    }
    return DFTU_OK;
}
