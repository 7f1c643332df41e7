// Coulomb integrals (mm'|m''m''') on the real-space grid (Sec. III; definition Eq. B2).
// The pair densities phi_c phi_d (c <= d) of one atom are placed on a zero-padded box around its sphere,
// all M(M+1)/2 of them at once; the Hartree potentials come from a 3-D discrete Fourier transform with the
// truncated Coulomb kernel 4 pi (1 - cos(G Rc)) / G^2 (2 pi Rc^2 at G = 0); (ab|cd) = dV sum_j phi_a(j)
// phi_b(j) v_cd(j).  Box edge >= 2R + Rc per axis rounded up to a 2,3,5-smooth size, Rc = 2R + 2 max(h):
// the potential inside the sphere is then free of periodic-image contributions.
//
// The transforms are the library's own: mixed-radix (5, 4, 3, 2) self-sorting Stockham passes over lines in
// shared memory, FP64, with the roots of unity tabulated once per transform length.  They are bound by the
// FP64 pipe, so the work is cut down:
//   - the kernel is real and even, so the potential of a real density is real: two pair densities share one
//     complex transform, as its real and imaginary parts;
//   - densities and the potentials wanted lie in the sphere's bounding box, about half the padded edge: lines
//     that are zero or not wanted are skipped (3.5 of 6 full passes are left);
//   - the last forward axis, the product with the kernel and the first inverse axis run in one kernel;
//   - butterflies use the factored forms of the short transforms, and the kernel is tabulated once on the
//     octant of non-negative frequencies.
// One d shell of radius 4.5 at h = 0.25 (75^3 box, 15 pair densities): 9.75 ms per call as full complex transforms
// of every pair density with the short transforms as plain sums, 1.11 ms now (kernels 9.2 -> 0.77 ms, of which
// the fused last axis 0.38).
#include <algorithm>
#include <cmath>
#include <vector>

#include "dftu_internal.cuh"

namespace dftu {

static int smooth235(int n) {
    for (int m = std::max(n, 1);; ++m) {
        int k = m;
        for (int p : {2, 3, 5})
            while (k % p == 0) k /= p;
        if (k == 1) return m;
    }
}

constexpr int FFT_MAXN = 512;     // longest transform (box edge) handled
constexpr int FFT_MAXSTAGES = 12;
struct FftPlan {
    int n;
    int nst;
    int radix[FFT_MAXSTAGES];
};

static bool make_plan(int n, FftPlan& p) {
    p.n = n;
    p.nst = 0;
    int m = n;
    for (int r : {5, 4, 3, 2})
        while (m % r == 0) {
            if (p.nst == FFT_MAXSTAGES) return false;
            p.radix[p.nst++] = r;
            m /= r;
        }
    return m == 1 && n <= FFT_MAXN;
}

// Transform lengths, the box of the sphere's points and the tables of one integral set.
struct Box {
    int n[3];            // padded box
    int e[3];            // extent of the sphere's points (their bounding box starts at the box origin)
    double h[3];
    double Rc;
    FftPlan plan[3];
    const double2* w[3]; // roots exp(-2 pi i k / n), one table per axis
    const double* K;     // kernel on the frequencies 0 .. n/2 of every axis
    __host__ __device__ int half(int a) const { return n[a] / 2 + 1; }
};

// Roots of unity of the three axes (blockIdx.y).
__global__ void k_fft_roots(Box B, double2* w0, double2* w1, double2* w2) {
    const int a = blockIdx.y, n = B.n[a];
    double2* w = a == 0 ? w0 : a == 1 ? w1 : w2;
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    double s, c;
    sincospi(-2.0 * (double)k / (double)n, &s, &c);
    w[k] = make_double2(c, s);
}

// The truncated Coulomb kernel on the octant of non-negative frequencies (it depends on |G| alone), divided by
// the number of box points (the transforms are unnormalised).
__global__ void k_coulomb_kernel(Box B, double* __restrict__ K) {
    const int hx = B.half(0), hy = B.half(1), hz = B.half(2);
    const int g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= hx * hy * hz) return;
    const int x = g % hx, y = (g / hx) % hy, z = g / (hx * hy);
    const double tpi = 6.283185307179586476925286766559;
    const double gx = tpi * x / (B.n[0] * B.h[0]), gy = tpi * y / (B.n[1] * B.h[1]), gz = tpi * z / (B.n[2] * B.h[2]);
    const double G2 = gx * gx + gy * gy + gz * gz;
    const double v = (g == 0) ? tpi * B.Rc * B.Rc : 2.0 * tpi * (1.0 - cos(sqrt(G2) * B.Rc)) / G2;   // 2 pi Rc^2 ; 4 pi (1-cos)/G^2
    K[g] = v / ((double)B.n[0] * B.n[1] * B.n[2]);
}

__device__ __forceinline__ double2 add2(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 sub2(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }
// a + i s b
__device__ __forceinline__ double2 addi(double2 a, double2 b, double s) { return make_double2(fma(-s, b.y, a.x), fma(s, b.x, a.y)); }

// Short transforms X_q = sum_r u_r exp(s 2 pi i q r / R), s = +-1, in place.
template <int R>
__device__ __forceinline__ void dft(double2 (&u)[R], double s);
template <>
__device__ __forceinline__ void dft<2>(double2 (&u)[2], double) {
    const double2 a = u[0];
    u[0] = add2(a, u[1]);
    u[1] = sub2(a, u[1]);
}
template <>
__device__ __forceinline__ void dft<3>(double2 (&u)[3], double s) {
    const double2 t = add2(u[1], u[2]), d = sub2(u[1], u[2]);
    const double2 m = make_double2(fma(-0.5, t.x, u[0].x), fma(-0.5, t.y, u[0].y));
    u[0] = add2(u[0], t);
    const double c = s * 0.86602540378443864676;   // sin(2 pi / 3)
    u[1] = addi(m, d, c);
    u[2] = addi(m, d, -c);
}
template <>
__device__ __forceinline__ void dft<4>(double2 (&u)[4], double s) {
    const double2 a = add2(u[0], u[2]), b = sub2(u[0], u[2]), c = add2(u[1], u[3]), d = sub2(u[1], u[3]);
    u[0] = add2(a, c);
    u[2] = sub2(a, c);
    u[1] = make_double2(b.x - s * d.y, b.y + s * d.x);
    u[3] = make_double2(b.x + s * d.y, b.y - s * d.x);
}
template <>
__device__ __forceinline__ void dft<5>(double2 (&u)[5], double s) {
    const double c1 = 0.30901699437494742410, c2 = -0.80901699437494742410;   // cos(2 pi / 5), cos(4 pi / 5)
    const double s1 = 0.95105651629515357212, s2 = 0.58778525229247312917;    // sin of the same
    const double2 t1 = add2(u[1], u[4]), t2 = add2(u[2], u[3]), t3 = sub2(u[1], u[4]), t4 = sub2(u[2], u[3]);
    const double2 m1 = make_double2(fma(c2, t2.x, fma(c1, t1.x, u[0].x)), fma(c2, t2.y, fma(c1, t1.y, u[0].y)));
    const double2 m2 = make_double2(fma(c1, t2.x, fma(c2, t1.x, u[0].x)), fma(c1, t2.y, fma(c2, t1.y, u[0].y)));
    const double2 n1 = make_double2(fma(s2, t4.x, s1 * t3.x), fma(s2, t4.y, s1 * t3.y));
    const double2 n2 = make_double2(fma(-s1, t4.x, s2 * t3.x), fma(-s1, t4.y, s2 * t3.y));
    u[0] = add2(u[0], add2(t1, t2));
    u[1] = addi(m1, n1, s);
    u[4] = addi(m1, n1, -s);
    u[2] = addi(m2, n2, s);
    u[3] = addi(m2, n2, -s);
}

// One radix-R pass over L lines of length n (line stride ld): p points are transformed already.
template <int R, int L>
__device__ __forceinline__ void fft_pass(const double2* src, double2* dst, const double2* w, int n, int ld, int p, double s) {
    const int T = n / R, step = n / (p * R);
    for (int e = threadIdx.x; e < T * L; e += blockDim.x) {
        const int l = e % L, i = e / L;
        const int k = i % p;
        double2 u[R];
#pragma unroll
        for (int r = 0; r < R; ++r) u[r] = src[l * ld + i + r * T];
        if (k)
#pragma unroll
            for (int r = 1; r < R; ++r) {   // times exp(s 2 pi i k r / (p R)); the table holds exp(-2 pi i j / n)
                const double2 t = w[k * r * step];
                const double ty = -s * t.y;
                u[r] = make_double2(u[r].x * t.x - u[r].y * ty, u[r].x * ty + u[r].y * t.x);
            }
        dft<R>(u, s);
        const int j = (i / p) * p * R + k;
#pragma unroll
        for (int r = 0; r < R; ++r) dst[l * ld + j + r * p] = u[r];
    }
}

// Transform of the L lines in buf[0] (s = -1 forward, +1 inverse, unnormalised); returns the buffer that holds
// the result.  Every thread of the CTA calls it; it starts and ends with a barrier.
template <int L>
__device__ __forceinline__ int fft_lines(double2* const (&buf)[2], int src, const double2* w, const FftPlan& plan, int ld, double s) {
    int p = 1;
    __syncthreads();
    for (int q = 0; q < plan.nst; ++q) {
        const int R = plan.radix[q];
        double2 *a = buf[src], *b = buf[1 - src];
        if (R == 5) fft_pass<5, L>(a, b, w, plan.n, ld, p, s);
        else if (R == 4) fft_pass<4, L>(a, b, w, plan.n, ld, p, s);
        else if (R == 3) fft_pass<3, L>(a, b, w, plan.n, ld, p, s);
        else fft_pass<2, L>(a, b, w, plan.n, ld, p, s);
        __syncthreads();
        src = 1 - src;
        p *= R;
    }
    return src;
}

// Lines of one axis.  The input line has nin values (the rest are zeros), the output keeps nout.  Line index
// = (outer index) * ninner + inner index; element (outer, inner, i) sits at outer * out_stride + inner + i * inner
// stride, for input and output arrays of their own shapes.
//   AXIS 0: contiguous lines (inner stride 1); AXIS 1, 2: adjacent lines are adjacent in memory.
// MUL: forward, product with the kernel, inverse (the last axis).
struct Lines {
    int64_t nlines;
    int ninner;            // lines adjacent in memory
    int nin, nout;
    int64_t in_outer, out_outer;
    int in_step, out_step; // between successive values of a line
};

template <int AXIS, int L, int MUL>
__global__ void __launch_bounds__(256) k_fft_lines(Box B, Lines q, const double2* in, double2* out, double s) {
    extern __shared__ double2 fft_smem[];
    const FftPlan& plan = B.plan[AXIS];
    const int n = plan.n, ld = n | 1;   // an odd stride keeps the L lines of one position in different banks
    double2* const buf[2] = {fft_smem, fft_smem + L * ld};
    double2* w = fft_smem + 2 * L * ld;
    const int64_t L0 = (int64_t)blockIdx.x * L;
    for (int k = threadIdx.x; k < n; k += blockDim.x) w[k] = B.w[AXIS][k];
    for (int e = threadIdx.x; e < n * L; e += blockDim.x) {
        const int l = AXIS == 0 ? e / n : e % L, i = AXIS == 0 ? e - l * n : e / L;
        const int64_t line = L0 + l;
        double2 x = make_double2(0.0, 0.0);
        if (line < q.nlines && i < q.nin) x = in[(line / q.ninner) * q.in_outer + (AXIS == 0 ? 0 : line % q.ninner) + (int64_t)i * q.in_step];
        buf[0][l * ld + i] = x;
    }
    int r = fft_lines<L>(buf, 0, w, plan, ld, s);
    if (MUL) {
        const int hx = B.half(0), hy = B.half(1);
        for (int e = threadIdx.x; e < n * L; e += blockDim.x) {
            const int l = e % L, z = e / L;
            const int64_t line = L0 + l;
            if (line < q.nlines) {
                const int xy = (int)(line % q.ninner), x = xy % B.n[0], y = xy / B.n[0];
                const double k = B.K[min(x, B.n[0] - x) + hx * (min(y, B.n[1] - y) + (int64_t)hy * min(z, n - z))];
                double2& v = buf[r][l * ld + z];
                v = make_double2(v.x * k, v.y * k);
            }
        }
        r = fft_lines<L>(buf, r, w, plan, ld, -s);
    }
    for (int e = threadIdx.x; e < q.nout * L; e += blockDim.x) {
        const int l = AXIS == 0 ? e / q.nout : e % L, i = AXIS == 0 ? e - l * q.nout : e / L;
        const int64_t line = L0 + l;
        if (line < q.nlines) out[(line / q.ninner) * q.out_outer + (AXIS == 0 ? 0 : line % q.ninner) + (int64_t)i * q.out_step] = buf[r][l * ld + i];
    }
}

// D[box][point] = phi_c phi_d + i phi_c' phi_d' for successive pairs c <= d (pair index in the order of the
// (c, d) loop) on the sphere's bounding box; lin[j] = the point's index there.
__global__ void k_scatter_pairs(const double* __restrict__ phi, const int* __restrict__ u, int64_t p0, int np, int M, int P,
                                int ux, int uy, int uz, int ex, int ey, int64_t E, double2* __restrict__ D, int* __restrict__ lin) {
    const int P2 = (P + 1) / 2;
    const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= (int64_t)np * P2) return;
    const int bx = (int)(g / np), j = (int)(g % np);
    const int64_t q = p0 + j;
    const int at = u[3 * q] - ux + ex * (u[3 * q + 1] - uy + ey * (u[3 * q + 2] - uz));
    const double* ph = phi + (int64_t)j * M;
    double v[2] = {0.0, 0.0};
    for (int t = 0; t < 2; ++t) {
        const int pcd = 2 * bx + t;
        if (pcd >= P) break;
        int c = 0, rem = pcd;
        while (rem >= M - c) { rem -= M - c; ++c; }
        v[t] = ph[c] * ph[c + rem];
    }
    D[(int64_t)bx * E + at] = make_double2(v[0], v[1]);
    if (bx == 0) lin[j] = at;
}

// W[ab][cd] = dV sum_j phi_a(j) phi_b(j) v_cd(j); one CTA per (ab, cd), fixed-order reduction.
__global__ void __launch_bounds__(CTA) k_pair_dot(const double* __restrict__ phi, const int* __restrict__ lin, int np, int M, int P,
                                                  const double2* __restrict__ D, int64_t E, double dV, double* __restrict__ W) {
    const int pab = blockIdx.x, pcd = blockIdx.y;
    int a = 0, rem = pab;
    while (rem >= M - a) { rem -= M - a; ++a; }
    const int b = a + rem;
    const double* v = reinterpret_cast<const double*>(D + (int64_t)(pcd / 2) * E) + (pcd & 1);
    __shared__ double red[CTA];
    double acc = 0.0;
#pragma unroll 8
    for (int j = threadIdx.x; j < np; j += CTA) {
        const double* ph = phi + (int64_t)j * M;
        acc = fma(ph[a] * ph[b], v[2 * lin[j]], acc);
    }
    red[threadIdx.x] = acc;
    __syncthreads();
    for (int s = CTA / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s) red[threadIdx.x] += red[threadIdx.x + s];
        __syncthreads();
    }
    if (threadIdx.x == 0) W[pab * P + pcd] = red[0] * dV;
}

__global__ void k_expand(const double* __restrict__ W, int M, int P, double* __restrict__ V) {
    int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= M * M * M * M) return;
    int a = e / (M * M * M), b = (e / (M * M)) % M, c = (e / M) % M, d = e % M;
    auto pidx = [M](int x, int y) {
        int lo = x < y ? x : y, hi = x < y ? y : x;
        return lo * M - lo * (lo - 1) / 2 + (hi - lo);
    };
    V[e] = W[pidx(a, b) * P + pidx(c, d)];
}

// One axis.  16 lines per CTA fill its 256 threads on the usual lengths (radix-5 butterflies of 75 points: 240
// of them); from 208 points on their two buffers would leave one CTA per SM, and 8 lines are taken.
template <int AXIS, int L, int MUL>
static cudaError_t run_lines(const Box& B, const Lines& q, const double2* in, double2* out, double s, cudaStream_t st) {
    const int n = B.n[AXIS];
    const int smem = (2 * L * (n | 1) + n) * (int)sizeof(double2);
    auto fn = k_fft_lines<AXIS, L, MUL>;
    cudaError_t e = cudaSuccess;
    if (smem > 48 * 1024 && !smem_configured((const void*)fn, smem)) e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    fn<<<(unsigned)((q.nlines + L - 1) / L), 256, smem, st>>>(B, q, in, out, s);
    return cudaGetLastError();
}

template <int AXIS, int MUL>
static cudaError_t lines(const Box& B, const Lines& q, const double2* in, double2* out, double s, cudaStream_t st) {
    return B.n[AXIS] < 208 ? run_lines<AXIS, 16, MUL>(B, q, in, out, s, st) : run_lines<AXIS, 8, MUL>(B, q, in, out, s, st);
}

// Potentials of P2 complex densities on the bounding box, D[P2][ez][ey][ex] in place.  X holds lines transformed
// along x ([P2][ez][ey][n0]), Y along x and y ([P2][ez][n1][n0]).
static cudaError_t poisson(const Box& B, int P2, double2* D, double2* X, double2* Y, cudaStream_t st) {
    const int n0 = B.n[0], n1 = B.n[1], ex = B.e[0], ey = B.e[1], ez = B.e[2];
    const int64_t n01 = (int64_t)n0 * n1;
    cudaError_t e = lines<0, 0>(B, Lines{(int64_t)P2 * ez * ey, 1, ex, n0, ex, n0, 1, 1}, D, X, -1.0, st);
    if (e == cudaSuccess) e = lines<1, 0>(B, Lines{(int64_t)P2 * ez * n0, n0, ey, n1, (int64_t)ey * n0, n01, n0, n0}, X, Y, -1.0, st);
    if (e == cudaSuccess) e = lines<2, 1>(B, Lines{P2 * n01, (int)n01, ez, ez, ez * n01, ez * n01, (int)n01, (int)n01}, Y, Y, -1.0, st);
    if (e == cudaSuccess) e = lines<1, 0>(B, Lines{(int64_t)P2 * ez * n0, n0, n1, ey, n01, (int64_t)ey * n0, n0, n0}, Y, X, 1.0, st);
    if (e == cudaSuccess) e = lines<0, 0>(B, Lines{(int64_t)P2 * ez * ey, 1, n0, ex, n0, ex, 1, 1}, X, D, 1.0, st);
    return e;
}

int coulomb_atom(const View& v, const Ctx& c, int atom, double* V_dev, std::string& err) {
    const dftu_atom& at = c.atoms[atom];
    const int M = c.M[atom];
    const int P = M * (M + 1) / 2;
    const double R = at.radius;
    const double hmax = std::max(c.grid.h[0], std::max(c.grid.h[1], c.grid.h[2]));
    const double Rc = 2.0 * R + 2.0 * hmax;
    Box B;
    B.Rc = Rc;
    for (int a = 0; a < 3; ++a) {
        B.h[a] = c.grid.h[a];
        B.n[a] = smooth235((int)std::ceil((2.0 * R + Rc) / c.grid.h[a]));
        if (!make_plan(B.n[a], B.plan[a])) {
            err = "coulomb: Poisson box edge " + std::to_string(B.n[a]) + " exceeds " + std::to_string(FFT_MAXN) + " points";
            return DFTU_ERR_INVALID_ARG;
        }
        B.e[a] = c.atom_umax[atom][a] - c.atom_umin[atom][a] + 1;   // at most 2R/h + 1 points, below the box edge
    }
    const int P2 = (P + 1) / 2;
    const int64_t E = (int64_t)B.e[0] * B.e[1] * B.e[2];
    const int np = c.npts[atom];
    const int64_t p0 = c.atom_p0[atom];
    const double* phi = v.phi64 + c.atom_phi0[atom];
    const int ux = c.atom_umin[atom][0], uy = c.atom_umin[atom][1], uz = c.atom_umin[atom][2];
    // Everything runs on a private stream with stream-ordered scratch: no device-wide synchronisation,
    // only this stream is waited for before the result is returned.
    cudaStream_t st = nullptr;
    cudaError_t e = cudaStreamCreateWithFlags(&st, cudaStreamNonBlocking);
    if (e != cudaSuccess) { cudaGetLastError(); err = std::string("coulomb: ") + cudaGetErrorString(e); return DFTU_ERR_CUDA; }
    // one scratch block: D, X, Y, the roots, the kernel octant, W, the points' indices
    const size_t nD = (size_t)P2 * E, nX = (size_t)P2 * B.e[2] * B.e[1] * B.n[0], nY = (size_t)P2 * B.e[2] * B.n[1] * B.n[0];
    const size_t nroot = (size_t)B.n[0] + B.n[1] + B.n[2], nK = (size_t)B.half(0) * B.half(1) * B.half(2);
    const size_t bytes = (nD + nX + nY + nroot) * sizeof(double2) + (nK + (size_t)P * P) * sizeof(double) + (size_t)np * sizeof(int);
    double2* D = nullptr;
    double* W = nullptr;
    e = cudaMallocAsync(reinterpret_cast<void**>(&D), bytes, st);
    if (e == cudaSuccess) {
        double2 *X = D + nD, *Y = X + nX, *w = Y + nY;
        double* K = reinterpret_cast<double*>(w + nroot);
        W = K + nK;
        int* lin = reinterpret_cast<int*>(W + (size_t)P * P);
        B.w[0] = w; B.w[1] = w + B.n[0]; B.w[2] = w + B.n[0] + B.n[1];
        B.K = K;
        const int nmax = std::max(B.n[0], std::max(B.n[1], B.n[2]));
        k_fft_roots<<<dim3((nmax + 127) / 128, 3), 128, 0, st>>>(B, w, w + B.n[0], w + B.n[0] + B.n[1]);
        e = cudaGetLastError();
        if (e == cudaSuccess) {
            k_coulomb_kernel<<<(unsigned)((nK + 127) / 128), 128, 0, st>>>(B, K);
            e = cudaGetLastError();
        }
        if (e == cudaSuccess) e = cudaMemsetAsync(D, 0, nD * sizeof(double2), st);
        if (e == cudaSuccess) {
            const int64_t work = (int64_t)np * P2;
            k_scatter_pairs<<<(unsigned)((work + 255) / 256), 256, 0, st>>>(phi, v.pt_u, p0, np, M, P, ux, uy, uz, B.e[0], B.e[1], E, D, lin);
            e = cudaGetLastError();
        }
        if (e == cudaSuccess) e = poisson(B, P2, D, X, Y, st);
        if (e == cudaSuccess) {
            k_pair_dot<<<dim3(P, P), CTA, 0, st>>>(phi, lin, np, M, P, D, E, v.dV, W);
            e = cudaGetLastError();
        }
    }
    if (e == cudaSuccess) {
        k_expand<<<(M * M * M * M + 255) / 256, 256, 0, st>>>(W, M, P, V_dev);
        e = cudaGetLastError();
    }
    if (D) cudaFreeAsync(D, st);
    cudaError_t es = cudaStreamSynchronize(st);
    if (e == cudaSuccess) e = es;
    cudaStreamDestroy(st);
    if (e != cudaSuccess) {
        cudaGetLastError();
        err = std::string("coulomb: ") + cudaGetErrorString(e);
        return e == cudaErrorMemoryAllocation ? DFTU_ERR_ALLOC : DFTU_ERR_CUDA;
    }
    return DFTU_OK;
}

}  // namespace dftu
