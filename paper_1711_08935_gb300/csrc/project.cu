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

// p[ks][band][moff_I + m] = sum over the atom's tiles of the tile partials, each image segment's sum times its Bloch
// phase.  One CTA per (k*spin, 32 bands, atom): eight warps take successive ranges of the atom's tiles, every lane
// one band with all M orbitals, so that M loads per tile and several tiles are in flight; the ranges are added in
// order and p is written with its orbitals adjacent.  An atom's tiles take successive slots, M apart.  (One thread per
// (state, orbital), walking the tiles: a chain of latencies, and p written 16 bytes at a time.  From cold caches, 48
// tiles per atom, 512 states, 64 orbitals: 45.8 -> 26.0 us; 64 atoms, 256 states: 37 -> 34 us.)
constexpr int RED_BANDS = 32, RED_SLICES = CTA / RED_BANDS, RED_LD = RED_BANDS + 1;

// acc += ph s, rounded alike in both forms of the reduce.
__device__ __forceinline__ void add_segment(double2& acc, double2 ph, double2 s) {
    acc.x = fma(ph.x, s.x, fma(-ph.y, s.y, acc.x));
    acc.y = fma(ph.x, s.y, fma(ph.y, s.x, acc.y));
}

template <int M>
__device__ __forceinline__ void reduce_atom(const View& v, int nbands, int ks, int a, int band0, int table, int64_t p_stride, double2* sm) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int t0 = v.atom_tile_beg[a], t1 = v.atom_tile_end[a];
    const int per = (t1 - t0 + RED_SLICES - 1) / RED_SLICES;
    const int tb = t0 + w * per, te = min(t1, tb + per);
    const bool in = band0 + lane < nbands;
    const double2* base = v.part + table * v.part_dir_stride + ((int64_t)ks * v.TM + v.tiles[t0].moff) * v.max_bands + band0 + lane;
    const double2* phk = v.seg_phase + ks / v.ns;
    double2 acc[M], s[M];
#pragma unroll
    for (int m = 0; m < M; ++m) acc[m] = s[m] = make_double2(0.0, 0.0);
    int seg = -1;
    double2 ph = make_double2(0.0, 0.0);
    auto flush = [&]() {
#pragma unroll
        for (int m = 0; m < M; ++m) {
            add_segment(acc[m], ph, s[m]);
            s[m] = make_double2(0.0, 0.0);
        }
    };
    constexpr int B = M <= 3 ? 4 : M == 5 ? 2 : 1;   // tiles in flight
    for (int t = tb; t < te; t += B) {
        double2 x[B][M];
        int sg[B];
#pragma unroll
        for (int u = 0; u < B; ++u) {
            const bool on = t + u < te;
            sg[u] = on ? v.tiles[t + u].seg : -1;
#pragma unroll
            for (int m = 0; m < M; ++m)
                x[u][m] = (on && in) ? base[((int64_t)(t + u - t0) * M + m) * v.max_bands] : make_double2(0.0, 0.0);
        }
#pragma unroll
        for (int u = 0; u < B; ++u) {
            if (t + u >= te) break;
            if (sg[u] != seg) {
                if (seg >= 0) flush();
                seg = sg[u];
                ph = phk[(int64_t)seg * v.nk];
            }
#pragma unroll
            for (int m = 0; m < M; ++m) { s[m].x += x[u][m].x; s[m].y += x[u][m].y; }
        }
    }
    if (seg >= 0) flush();
#pragma unroll
    for (int m = 0; m < M; ++m) sm[(w * M + m) * RED_LD + lane] = acc[m];
    __syncthreads();
    const int used = min(RED_SLICES, (t1 - t0 + per - 1) / per);
    for (int e = threadIdx.x; e < M * RED_BANDS; e += CTA) {
        const int b = e / M, m = e - b * M;
        if (band0 + b >= nbands) break;
        double re = 0.0, im = 0.0;
        for (int q = 0; q < used; ++q) {
            const double2 y = sm[(q * M + m) * RED_LD + b];
            re += y.x;
            im += y.y;
        }
        re *= v.dV;
        im *= v.dV;
        if (!isfinite(re) || !isfinite(im)) atomicOr(v.status, ST_NONFINITE);
        v.p[table * p_stride + ((int64_t)ks * v.max_bands + band0 + b) * v.MT + v.atom_moff[a] + m] = make_double2(re, im);
    }
}

// CTAs of one system's reduce: (k*spin, band chunk, atom), atoms fastest.
__host__ __device__ static int64_t reduce_ctas(const View& v, int nbands) { return (int64_t)v.nk * v.ns * ((nbands + RED_BANDS - 1) / RED_BANDS) * v.natoms; }

__device__ __forceinline__ void reduce_item(const View& v, int nbands, int64_t id, int table, int64_t p_stride) {
    __shared__ double2 sm[RED_SLICES * MAXM * RED_LD];
    const int chunks = (nbands + RED_BANDS - 1) / RED_BANDS;
    if (id >= (int64_t)v.nk * v.ns * chunks * v.natoms) return;
    const int a = (int)(id % v.natoms);
    const int64_t r = id / v.natoms;
    const int ks = (int)(r / chunks), band0 = (int)(r % chunks) * RED_BANDS;
    switch (v.atom_M[a]) {
        case 1: reduce_atom<1>(v, nbands, ks, a, band0, table, p_stride, sm); break;
        case 3: reduce_atom<3>(v, nbands, ks, a, band0, table, p_stride, sm); break;
        case 5: reduce_atom<5>(v, nbands, ks, a, band0, table, p_stride, sm); break;
        default: reduce_atom<7>(v, nbands, ks, a, band0, table, p_stride, sm); break;
    }
}

__global__ void __launch_bounds__(CTA, 2) k_tile_reduce(View v, int nbands) {
    dependent_release();
    dependent_wait();
    reduce_item(v, nbands, blockIdx.x, 0, 0);
}

// The same sums with a thread per (k*spin, orbital, band), band fastest, walking the atom's tiles in order.  Where the
// form above takes more than two waves, the SMs are full either way and this one holds more warps: 512 CTAs of the form
// above 37 (this) against 33 us, 1024 CTAs 31 against 40, 2048 CTAs 64 against 84.  (In the ranges of the form above,
// for one order at every size, it is bound by the instructions that close them: 64 atoms, 2048 states 100 -> 130 us.)
__device__ __forceinline__ void reduce_state(const View& v, int nbands, int64_t g) {
    if (g >= (int64_t)v.nk * v.ns * v.MT * nbands) return;
    const int band = (int)(g % nbands), j = (int)(g / nbands % v.MT), ks = (int)(g / nbands / v.MT);
    const int a = v.orb_atom[j], m = j - v.atom_moff[a];
    const double2* part = v.part + ((int64_t)ks * v.TM + m) * v.max_bands + band;
    const double2* phase = v.seg_phase + ks / v.ns;
    double2 sum = make_double2(0.0, 0.0), in_seg = sum;
    int seg = -1;
    for (int t = v.atom_tile_beg[a]; t < v.atom_tile_end[a]; ++t) {
        const Tile& tl = v.tiles[t];
        if (tl.seg != seg) {
            if (seg >= 0) add_segment(sum, phase[(int64_t)seg * v.nk], in_seg);
            seg = tl.seg;
            in_seg = make_double2(0.0, 0.0);
        }
        const double2 x = part[(int64_t)tl.moff * v.max_bands];
        in_seg.x += x.x;
        in_seg.y += x.y;
    }
    add_segment(sum, phase[(int64_t)seg * v.nk], in_seg);
    sum.x *= v.dV;
    sum.y *= v.dV;
    if (!isfinite(sum.x) || !isfinite(sum.y)) atomicOr(v.status, ST_NONFINITE);
    v.p[((int64_t)ks * v.max_bands + band) * v.MT + j] = sum;
}

__global__ void k_tile_reduce_states(View v, int nbands) {
    dependent_release();
    dependent_wait();
    reduce_state(v, nbands, (int64_t)blockIdx.x * blockDim.x + threadIdx.x);
}

// The tables of the current (blockIdx.y) in one launch, each into its slice of p.
__global__ void __launch_bounds__(CTA, 2) k_tile_reduce_tables(View v, int nbands, int64_t p_stride) {
    if ((int)blockIdx.y < cur_tables(v.atom_M[blockIdx.x % v.natoms])) reduce_item(v, nbands, blockIdx.x, blockIdx.y, p_stride);
}

// Every member in the form that the same call made alone takes (states_above: reduce_by_states), so that it gets the same bits.
__global__ void __launch_bounds__(CTA, 2) k_tile_reduce_batch(const View* __restrict__ views, const ProjArgs* __restrict__ args, int64_t states_above) {
    const View& v = views[blockIdx.y];
    const int nbands = args[blockIdx.y].nbands;
    if (reduce_ctas(v, nbands) > states_above) reduce_state(v, nbands, (int64_t)blockIdx.x * CTA + threadIdx.x);
    else reduce_item(v, nbands, blockIdx.x, 0, 0);
}

// The thread-per-state form above this many CTAs of the other: two waves (two CTAs per SM).
static int64_t reduce_by_states() { return 4 * (int64_t)sm_count(); }

int64_t tile_reduce_blocks(const View& v, int nbands) {
    const int64_t ctas = reduce_ctas(v, nbands);
    return ctas > reduce_by_states() ? ((int64_t)v.nk * v.ns * v.MT * nbands + CTA - 1) / CTA : ctas;
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
        else e = run_project<P_PAIR, 8, 8, 8, 5, 2, 1, 1, CTA, TILE, false, true>(v, a, st);
    } else if (prec == DFTU_C64) {
        e = project_f32(v, a, variant, st, &vp);
    } else if (mode == DFTU_F64_NATIVE) {
        e = run_project<P_F64, 8, 1, 4, 0>(v, a, st);
    } else {
        e = project_pair(v, a, variant, st, &vp);
    }
    if (e != cudaSuccess) return e;
    return launch_tile_reduce(vp, nbands, st);
}

cudaError_t launch_project_c64_tiles(const View& sub, const void* psi, int nbands, int64_t sk, int64_t ss, int64_t sn,
                                     cudaStream_t st) {
    ProjArgs a{psi, sk, ss, sn, nbands};
    return project_f32(sub, a, 0, st, nullptr);
}

cudaError_t launch_tile_reduce(const View& v, int nbands, cudaStream_t st) {
    auto fn = reduce_ctas(v, nbands) > reduce_by_states() ? k_tile_reduce_states : k_tile_reduce;
    return launch_dependent(fn, (unsigned)tile_reduce_blocks(v, nbands), CTA, 0, st, v, nbands);
}

cudaError_t launch_project_dirs(const View& v, const void* psi, dftu_prec prec, dftu_f64_mode mode, int nbands,
                                int64_t sk, int64_t ss, int64_t sn, bool gauge, double2* p_out, int64_t p_stride,
                                cudaStream_t st) {
    ProjArgs a{psi, sk, ss, sn, nbands};
    cudaError_t e;
    // the fixed shapes of the gauge path, with and without the phases
    if (prec == DFTU_C64) e = gauge ? run_project<P_F32, 8, 16, 8, 0, 2, 1, 3>(v, a, st) : run_project<P_F32, 8, 16, 8, 0, 2, 0, 3>(v, a, st);
    else if (mode == DFTU_F64_NATIVE) e = gauge ? run_project<P_F64, 8, 1, 4, 0, 2, 1, 3>(v, a, st) : run_project<P_F64, 8, 1, 4, 0, 2, 0, 3>(v, a, st);
    else e = gauge ? run_project<P_PAIR, 8, 8, 8, 5, 2, 1, 3, CTA, TILE, false, true>(v, a, st) : run_project<P_PAIR, 8, 8, 8, 5, 2, 0, 3, CTA, TILE, false, true>(v, a, st);
    if (e != cudaSuccess) return e;
    View vd = v;
    vd.p = p_out;
    k_tile_reduce_tables<<<dim3((unsigned)reduce_ctas(v, nbands), 3), CTA, 0, st>>>(vd, nbands, p_stride);
    return cudaGetLastError();
}

cudaError_t launch_project_batch(const BatchLaunch& b, dftu_prec prec, dftu_f64_mode mode, int variant, cudaStream_t st) {
    cudaError_t e;
    if (prec == DFTU_C64) e = project_f32_batch(b, variant, st);
    else if (mode == DFTU_F64_NATIVE) e = run_project_batch<P_F64, 8, 1, 4, 0>(b, st);
    else e = project_pair_batch(b, variant, st);
    if (e != cudaSuccess) return e;
    k_tile_reduce_batch<<<dim3((unsigned)b.max_reduce_ctas, b.nsys), CTA, 0, st>>>(b.views, b.args, reduce_by_states());
    return cudaGetLastError();
}

}  // namespace dftu
