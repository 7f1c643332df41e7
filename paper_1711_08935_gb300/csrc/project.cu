// Launches of the projection (kernels in project_kernels.cuh) and of the tile reduce that completes it.
#include <mutex>
#include <utility>

#include "project_kernels.cuh"

namespace dftu {

// One record per (kernel, device): the largest dynamic shared memory size already allowed.
bool smem_configured(const void* fn, int bytes) {
    static std::mutex mu;
    static std::vector<std::pair<std::pair<const void*, int>, int>> done;
    int dev = 0;
    cudaGetDevice(&dev);
    std::lock_guard<std::mutex> lock(mu);
    for (auto& d : done)
        if (d.first.first == fn && d.first.second == dev) {
            if (d.second >= bytes) return true;
            d.second = bytes;
            return false;
        }
    done.push_back({{fn, dev}, bytes});
    return false;
}

// p[ks][band][moff_I + m] = sum over the atom's tiles (fixed order) of the tile partials; one thread per
// (k*spin, orbital slot, band), band fastest.  An atom's tiles take successive slots, so the partials are read
// eight at a time, independently of the tile list: the sum is a chain of memory latencies otherwise
// (48 tiles per atom, 512 states, 64 orbitals: 45.8 us one at a time, 38.6 eight at a time, from cold caches).
__device__ __forceinline__ void tile_reduce_elem(const View& v, int nbands, int64_t g) {
    if (g >= (int64_t)v.nk * v.ns * v.MT * nbands) return;
    const int band = (int)(g % nbands);
    const int64_t r = g / nbands;
    const int j = (int)(r % v.MT);
    const int ks = (int)(r / v.MT);
    const int a = v.orb_atom[j];
    const int m = j - v.atom_moff[a];
    const int t0 = v.atom_tile_beg[a], t1 = v.atom_tile_end[a];
    const int64_t step = (int64_t)v.atom_M[a] * v.max_bands;   // from one tile's partial to the next tile's
    const double2* pr = v.part + ((int64_t)ks * v.TM + v.tiles[t0].moff + m) * v.max_bands + band;
    const double2* phk = v.seg_phase + ks / v.ns;
    // tiles of one image segment are consecutive: sum them, then apply that segment's Bloch phase
    double re = 0.0, im = 0.0, sr = 0.0, si = 0.0;
    int seg = v.tiles[t0].seg;
    double2 ph = phk[(int64_t)seg * v.nk];
    constexpr int B = 8;
    for (int t = t0; t < t1; t += B) {
        double2 x[B];
        int sg[B];
#pragma unroll
        for (int u = 0; u < B; ++u) {
            const bool in = t + u < t1;
            x[u] = in ? pr[(int64_t)(t + u - t0) * step] : make_double2(0.0, 0.0);
            sg[u] = in ? v.tiles[t + u].seg : -1;
        }
#pragma unroll
        for (int u = 0; u < B; ++u) {
            if (t + u >= t1) break;
            if (sg[u] != seg) {
                re += ph.x * sr - ph.y * si;
                im += ph.x * si + ph.y * sr;
                seg = sg[u];
                ph = phk[(int64_t)seg * v.nk];
                sr = si = 0.0;
            }
            sr += x[u].x;
            si += x[u].y;
        }
    }
    re += ph.x * sr - ph.y * si;
    im += ph.x * si + ph.y * sr;
    re *= v.dV;
    im *= v.dV;
    if (!isfinite(re) || !isfinite(im)) atomicOr(v.status, ST_NONFINITE);
    v.p[((int64_t)ks * v.max_bands + band) * v.MT + j] = make_double2(re, im);
}

__global__ void k_tile_reduce(View v, int nbands) {
    tile_reduce_elem(v, nbands, (int64_t)blockIdx.x * blockDim.x + threadIdx.x);
}

__global__ void k_tile_reduce_batch(const View* __restrict__ views, const ProjArgs* __restrict__ args) {
    tile_reduce_elem(views[blockIdx.y], args[blockIdx.y].nbands, (int64_t)blockIdx.x * blockDim.x + threadIdx.x);
}

// Whether MINB CTAs of fn with smem bytes of dynamic shared memory fit on one SM (cached per kernel and size).
bool fits_per_sm(const void* fn, int nt, size_t smem, int minb) {
    static std::mutex mu;
    static std::vector<std::pair<std::pair<const void*, size_t>, bool>> seen;
    std::lock_guard<std::mutex> lock(mu);
    for (auto& s : seen)
        if (s.first.first == fn && s.first.second == smem) return s.second;
    int n = 0;
    // the attribute only ever grows (smem_configured keeps the largest size set), so a smaller system
    // asked about later cannot leave it below what an earlier launch configured
    cudaError_t e = cudaSuccess;
    if (!smem_configured(fn, (int)smem)) e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess || cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, fn, nt, smem) != cudaSuccess) {
        cudaGetLastError();
        n = 0;
    }
    seen.push_back({{fn, smem}, n >= minb});
    return n >= minb;
}

int sm_count() {
    static std::mutex mu;
    static std::vector<std::pair<int, int>> seen;   // (device, SMs)
    int dev = 0;
    cudaGetDevice(&dev);
    std::lock_guard<std::mutex> lock(mu);
    for (auto& s : seen)
        if (s.first == dev) return s.second;
    int n = 1;
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    seen.push_back({dev, n});
    return n;
}

cudaError_t launch_project(const View& v, const void* psi, dftu_prec prec, dftu_f64_mode mode, int nbands,
                           int64_t sk, int64_t ss, int64_t sn, int variant, cudaStream_t st, bool gauge) {
    ProjArgs a{psi, sk, ss, sn, nbands};
    cudaError_t e;
    View vp = v;   // the View the projection ran with: its tiling feeds the tile reduce
    if (gauge) {   // one shape per arithmetic policy with the gauge phases (Sec. V)
        if (prec == DFTU_C64) e = run_project<P_F32, 8, 16, 8, 0, 2, 1>(v, a, st);
        else if (mode == DFTU_F64_NATIVE) e = run_project<P_F64, 8, 1, 4, 0, 2, 1>(v, a, st);
        else e = run_project<P_PAIR, 8, 8, 8, 5, 2, 1>(v, a, st);
    } else if (prec == DFTU_C64) {
        e = project_f32(v, a, variant, st, &vp);
    } else if (mode == DFTU_F64_NATIVE) {
        e = run_project<P_F64, 8, 1, 4, 0>(v, a, st);
    } else {
        e = project_pair(v, a, variant, st, &vp);
    }
    if (e != cudaSuccess) return e;
    int64_t n = (int64_t)v.nk * v.ns * nbands * v.MT;
    k_tile_reduce<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(vp, nbands);
    return cudaGetLastError();
}

cudaError_t launch_project_c64_tiles(const View& sub, const void* psi, int nbands, int64_t sk, int64_t ss, int64_t sn,
                                     cudaStream_t st) {
    ProjArgs a{psi, sk, ss, sn, nbands};
    return project_f32(sub, a, 0, st, nullptr);
}

cudaError_t launch_tile_reduce(const View& v, int nbands, cudaStream_t st) {
    int64_t n = (int64_t)v.nk * v.ns * nbands * v.MT;
    k_tile_reduce<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(v, nbands);
    return cudaGetLastError();
}

cudaError_t launch_project_dirs(const View& v, const void* psi, dftu_prec prec, dftu_f64_mode mode, int nbands,
                                int64_t sk, int64_t ss, int64_t sn, bool gauge, double2* p_out, int64_t p_stride,
                                cudaStream_t st) {
    ProjArgs a{psi, sk, ss, sn, nbands};
    cudaError_t e;
    // the fixed shapes of the gauge path, with and without the phases
    if (prec == DFTU_C64) e = gauge ? run_project<P_F32, 8, 16, 8, 0, 2, 1, 3>(v, a, st) : run_project<P_F32, 8, 16, 8, 0, 2, 0, 3>(v, a, st);
    else if (mode == DFTU_F64_NATIVE) e = gauge ? run_project<P_F64, 8, 1, 4, 0, 2, 1, 3>(v, a, st) : run_project<P_F64, 8, 1, 4, 0, 2, 0, 3>(v, a, st);
    else e = gauge ? run_project<P_PAIR, 8, 8, 8, 5, 2, 1, 3>(v, a, st) : run_project<P_PAIR, 8, 8, 8, 5, 2, 0, 3>(v, a, st);
    if (e != cudaSuccess) return e;
    int64_t n = (int64_t)v.nk * v.ns * nbands * v.MT;
    for (int d = 0; d < 3; ++d) {
        View vd = v;
        vd.part = v.part + d * v.part_dir_stride;
        vd.p = p_out + d * p_stride;
        k_tile_reduce<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(vd, nbands);
        e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t launch_project_batch(const BatchLaunch& b, dftu_prec prec, dftu_f64_mode mode, int variant, cudaStream_t st) {
    cudaError_t e;
    if (prec == DFTU_C64) e = project_f32_batch(b, variant, st);
    else if (mode == DFTU_F64_NATIVE) e = run_project_batch<P_F64, 8, 1, 4, 0>(b, st);
    else e = project_pair_batch(b, variant, st);
    if (e != cudaSuccess) return e;
    dim3 grid((unsigned)((b.max_reduce + 255) / 256), b.nsys);
    k_tile_reduce_batch<<<grid, 256, 0, st>>>(b.views, b.args);
    return cudaGetLastError();
}

}  // namespace dftu
