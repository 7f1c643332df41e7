// Gauge-invariant Hubbard operator and Hubbard current under a uniform vector potential A (Sec. V).
//
// Eq. (16) attaches the phase exp(-i A.r) to every localised orbital.  Measured from the atom the
// orbital belongs to (d = r - R_I, the atom-relative reading of Eq. 16), the projector becomes
//   p^A_m = <phi_m exp(-i A.d)|psi> = dV sum_j phi_m(j) exp(+i A.d_j) exp(+i k.T_j) psi(idx_j),
// and the operator scatters with exp(-i A.d_j).  The per-point phases are tabulated here once per A;
// the streaming kernels rotate each loaded state value (projection) or each update (apply) by them.
//
// Eq. (17), the Hubbard contribution to the current, is taken as J = sum w f <psi| -i [r, V_U^A] |psi>
// (the factor i of the velocity operator restored, since <[r, V]> + c.c. of a Hermitian V vanishes).
// With q^{(a)}_m = <phi_m d_a exp(-i A.d)|psi>, the projections onto orbitals weighted by the a-th
// displacement component (formed from the projections onto harmonics, View::phid64),
//   J_a = -i sum w f sum_{mm'} V_{mm'} [conj(q_m) p_m' - conj(p_m) q_m'],
// a real number; it equals dE_U/dA at fixed states.
#include "dftu_internal.cuh"

namespace dftu {

__device__ __forceinline__ void displacement(const View& v, int64_t j, int atom, double& dx, double& dy, double& dz) {
    const int ix = v.pt_u[3 * j], jy = v.pt_u[3 * j + 1], kz = v.pt_u[3 * j + 2];
    dx = __dsub_rn(__dadd_rn(__dmul_rn((double)ix, v.h0), v.o0), v.atom_pos[3 * atom]);
    dy = __dsub_rn(__dadd_rn(__dmul_rn((double)jy, v.h1), v.o1), v.atom_pos[3 * atom + 1]);
    dz = __dsub_rn(__dadd_rn(__dmul_rn((double)kz, v.h2), v.o2), v.atom_pos[3 * atom + 2]);
}

// exp(+i A.d_j) for every sphere point: FP64 (cos, sin) and the FP32 pair split (hi, hi, lo, lo).  The phase is a
// product over the axes, so a tile needs one FP64 sine and cosine per grid line it touches on each axis (tables in
// shared memory) and two complex products per point, instead of a sine and cosine per point, which the FP64 pipe
// bounds: 171 k points, 23.7 -> 13.4 us.  Now a chain of latencies (48 bytes written per point are 1.2 us of it).
constexpr int GAUGE_TAB = 256;   // grid lines per axis the tables hold; larger tiles evaluate every point
__global__ void __launch_bounds__(TILE) k_gauge_phases(View v, const double* __restrict__ A) {
    __shared__ double2 tab[3][GAUGE_TAB];
    __shared__ int lo[3], hi[3];
    if (blockIdx.x == 0 && threadIdx.x < 3) v.gaugeA[threadIdx.x] = A[threadIdx.x];   // for the real-time step
    const Tile t = v.tiles[blockIdx.x];
    const int i = threadIdx.x;
    if (i < 3) { lo[i] = 1 << 30; hi[i] = -(1 << 30); }
    __syncthreads();
    const int64_t j = t.p0 + i;
    int u[3] = {0, 0, 0};
    if (i < t.np)
        for (int a = 0; a < 3; ++a) {
            u[a] = v.pt_u[3 * j + a];
            atomicMin(&lo[a], u[a]);
            atomicMax(&hi[a], u[a]);
        }
    __syncthreads();
    const double h[3] = {v.h0, v.h1, v.h2}, o[3] = {v.o0, v.o1, v.o2};
    const bool small = hi[0] - lo[0] < GAUGE_TAB && hi[1] - lo[1] < GAUGE_TAB && hi[2] - lo[2] < GAUGE_TAB;
    if (small) {
        for (int e = i; e < 3 * GAUGE_TAB; e += TILE) {
            const int a = e / GAUGE_TAB, x = lo[a] + e % GAUGE_TAB;
            if (x > hi[a]) continue;
            const double d = __dsub_rn(__dadd_rn(__dmul_rn((double)x, h[a]), o[a]), v.atom_pos[3 * t.atom + a]);
            double s, c;
            sincos(A[a] * d, &s, &c);
            tab[a][e % GAUGE_TAB] = make_double2(c, s);
        }
        __syncthreads();
    }
    if (i >= t.np) return;
    double s, c;
    if (small) {
        const double2 x = tab[0][u[0] - lo[0]], y = tab[1][u[1] - lo[1]], z = tab[2][u[2] - lo[2]];
        const double2 xy = make_double2(x.x * y.x - x.y * y.y, x.x * y.y + x.y * y.x);
        c = xy.x * z.x - xy.y * z.y;
        s = xy.x * z.y + xy.y * z.x;
    } else {
        double dx, dy, dz;
        displacement(v, j, t.atom, dx, dy, dz);
        sincos(fma(A[2], dz, fma(A[1], dy, A[0] * dx)), &s, &c);
    }
    v.gauge_d[j] = make_double2(c, s);
    const float ch = __double2float_rn(c), sh = __double2float_rn(s);
    v.gauge_f[j] = make_float4(ch, sh, __double2float_rn(c - (double)ch), __double2float_rn(s - (double)sh));
}

cudaError_t launch_gauge_phases(const View& v, const double* A, cudaStream_t st) {
    k_gauge_phases<<<v.ntiles, TILE, 0, st>>>(v, A);
    return cudaGetLastError();
}

// Jpart[atom][z][a] = mult sum over the states of split z of w f Im sum_x conj(q^a_x) t_x, t = (V + V^+) p, which is
// Im sum_xy V_xy [conj(q_x) p_y - conj(p_x) q_y] for any V (occupation sums that a caller imports need not be
// Hermitian).  With q^a_x = sum_f A[f][a][x] P_f, P the projections onto the tables of the current, it is
// sum_(f, x) A[f][a][x] Im conj(P_f) t_x: one pass over a state's projections serves the three directions.  Collinear or
// unpolarised states.
// An atom's states are split over CUR_SPLIT CTAs, and a CTA takes CUR_STATES states at a time, a lane each; its four
// warps share the rows of t (through shared memory) and the functions f.  Few states, few warps: the FP64 pipe of one
// SM quarter, 80 cycles an instruction of a warp, would bound a thread per state.  16 atoms, 192 states: 12.8 us from
// cold caches (12.3 for the monomials with a thread per state, 60 % of the operations; 19.3 for the displaced orbitals).
constexpr int CUR_STATES = 32, CUR_PARTS = 4;

template <int M>
__device__ __forceinline__ void current_states(const View& v, const double* __restrict__ f, int nbands, int atom, int z,
                                               const double2* s_H, const double* s_A, double2* s_t, double (&acc)[3]) {
    constexpr int NF = cur_functions(M);
    const int lane = threadIdx.x % CUR_STATES, part = threadIdx.x / CUR_STATES;
    const int64_t slice = (int64_t)v.nk * v.ns * v.max_bands * v.MT;
    const int total = v.nk * v.ns * nbands;
    for (int e0 = z * CUR_STATES; e0 < total; e0 += CUR_SPLIT * CUR_STATES) {
        const bool in = e0 + lane < total;
        const int e = in ? e0 + lane : 0;
        const int ks = e / nbands, band = e % nbands, k = ks / v.ns, s = ks % v.ns;
        const double w = in ? v.wk[k] * f[(int64_t)ks * nbands + band] : 0.0;
        const int64_t row = ((int64_t)ks * v.max_bands + band) * v.MT + v.atom_moff[atom];
        double2 p[M];
#pragma unroll
        for (int x = 0; x < M; ++x) p[x] = v.p[row + x];
        __syncthreads();   // the states before have been read
        for (int x = part; x < M; x += CUR_PARTS) {
            double2 t = make_double2(0.0, 0.0);
#pragma unroll
            for (int y = 0; y < M; ++y) {
                const double2 H = s_H[s * M * M + x * M + y];
                t.x = fma(H.x, p[y].x, fma(-H.y, p[y].y, t.x));
                t.y = fma(H.x, p[y].y, fma(H.y, p[y].x, t.y));
            }
            s_t[x * CUR_STATES + lane] = t;
        }
        __syncthreads();
        double im[3] = {0.0, 0.0, 0.0};
        for (int q = part; q < NF; q += CUR_PARTS) {
            const double2 P = v.pgrad[(q / M) * slice + row + q % M];
#pragma unroll
            for (int x = 0; x < M; ++x) {
                const double2 t = s_t[x * CUR_STATES + lane];
                const double c = fma(P.x, t.y, -P.y * t.x);
#pragma unroll
                for (int a = 0; a < 3; ++a) im[a] = fma(s_A[(q * 3 + a) * MAXM + x], c, im[a]);
            }
        }
        if (in)   // (a state of weight zero may hold anything)
            for (int a = 0; a < 3; ++a) acc[a] = fma(w, im[a], acc[a]);
    }
}

__global__ void __launch_bounds__(CUR_STATES * CUR_PARTS) k_current(View v, const double* __restrict__ f, int nbands, double* __restrict__ Jpart) {
    const int atom = blockIdx.x, z = blockIdx.y;
    const int M = v.atom_M[atom];
    __shared__ double2 s_H[2 * MAXM * MAXM], s_t[MAXM * CUR_STATES];
    __shared__ double s_A[CUR_MAXF * 3 * MAXM];
    __shared__ double red[3][CUR_PARTS];
    const double2* V = v.V + v.atom_mat_off[atom];
    for (int e = threadIdx.x; e < v.ns * M * M; e += blockDim.x) {
        const int x = e / M % M, y = e % M;
        const double2 a = V[e], b = V[e - x * M - y + y * M + x];
        s_H[e] = make_double2(a.x + b.x, a.y - b.y);
    }
    for (int e = threadIdx.x; e < CUR_MAXF * 3 * MAXM; e += blockDim.x) s_A[e] = v.cur_A[(int64_t)atom * CUR_MAXF * 3 * MAXM + e];
    __syncthreads();
    double acc[3] = {0.0, 0.0, 0.0};
    switch (M) {
        case 1: current_states<1>(v, f, nbands, atom, z, s_H, s_A, s_t, acc); break;
        case 3: current_states<3>(v, f, nbands, atom, z, s_H, s_A, s_t, acc); break;
        case 5: current_states<5>(v, f, nbands, atom, z, s_H, s_A, s_t, acc); break;
        default: current_states<7>(v, f, nbands, atom, z, s_H, s_A, s_t, acc); break;
    }
    for (int a = 0; a < 3; ++a) {
        for (int off = 16; off > 0; off >>= 1) acc[a] += __shfl_xor_sync(0xffffffffu, acc[a], off);
        if ((threadIdx.x & 31) == 0) red[a][threadIdx.x >> 5] = acc[a];
    }
    __syncthreads();
    if (threadIdx.x < 3) {
        const double* r = red[threadIdx.x];
        Jpart[((int64_t)atom * CUR_SPLIT + z) * 3 + threadIdx.x] = ((v.ns == 1) ? 2.0 : 1.0) * (r[0] + r[1] + r[2] + r[3]);
    }
}

cudaError_t launch_current(const View& v, const double* f, int nbands, double* Jpart, cudaStream_t st) {
    k_current<<<dim3(v.natoms, CUR_SPLIT), CUR_STATES * CUR_PARTS, 0, st>>>(v, f, nbands, Jpart);
    return cudaGetLastError();
}

}  // namespace dftu
