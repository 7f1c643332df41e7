// Sphere gather + projection p = dV sum_j phi_m(j) exp(+i k.T_j) psi(idx_j)   (inside Eqs. 4 and 6).
//
// Work decomposition: one CTA per (tile, band chunk, k*spin).  A tile holds up to TILE points of one
// (atom, lattice image) segment, so its Bloch phase is a single number.  The CTA stages the tile's
// grid indices and orbital values in shared memory once and streams the bands of its chunk: Q
// adjacent lanes walk the points of one band (Q*16 or Q*8 contiguous bytes per band row when the
// points run along x), 32/Q bands per warp.  Partial sums per tile are written in FP64 without the
// phase; k_tile_reduce sums the tiles of each atom in a fixed order, applies each image segment's
// phase once and scales by dV, so results are deterministic.
//
// Arithmetic policies
//   F64  : complex128 states, FP64 FMAs (the FP64 pipe of this GPU runs at ~1/70 of FP32).
//   PAIR : complex128 states carried as pairs of FP32 numbers.  Each double is split (integer ops,
//          47 significant bits) into hi + lo floats scaled by 2^-Emax of its chain; products accumulate
//          into an accumulator offset by a power of two C >= 4*sum|terms| so that the running sum
//          moves in one binade: t = s - acc is exact and the rounding residual a*b - t is caught
//          in a second float.  Chains are merged with TwoSum.  Accuracy ~2^-44 of the chain scale.
//   F32  : complex64 states, FP32 orbitals hi + lo paired two orbitals at a time, FP32 chunk sums
//          merged with TwoSum per lane, FP64 across tiles.
#pragma once

#include <algorithm>

#include "dftu_internal.cuh"

namespace dftu {

// ------------------------------------------------------------------------------------------------
// small helpers
// ------------------------------------------------------------------------------------------------
__device__ __forceinline__ float2 ffma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 fadd2(float2 a, float2 b) { return __fadd2_rn(a, b); }

struct DF2 { float2 h, l; };   // (re, im) pair of double-float numbers

// Gather of one complex64 state value, 0 where !in (predicated, no branch).  The 64-byte prefetch size makes
// L2 fetch the 64-byte blocks that hold a run of points instead of whole 128-byte lines (1.31x instead of
// 1.64x the points' bytes on the oxide): this kernel is bound by that traffic, 330 -> 271 us for 512 oxide
// rows.  The complex128 projection, bound by its arithmetic and latency, ran no faster with it (587 -> 609 us,
// tile reduce included: the rest of the line is what the next lanes read) and keeps plain loads.
__device__ __forceinline__ float2 ld_gather(const float2* p, bool in) {
    float2 r = make_float2(0.f, 0.f);
    asm("{ .reg .pred q; setp.ne.b32 q, %3, 0; @q ld.global.nc.L1::no_allocate.L2::64B.v2.f32 {%0, %1}, [%2]; }"
        : "+f"(r.x), "+f"(r.y) : "l"(p), "r"((int)in));
    return r;
}

// Ask L2 to start fetching a line a later chain will read (no register is held for it).
__device__ __forceinline__ void prefetch_l2(const void* ptr) { asm volatile("prefetch.global.L2 [%0];" ::"l"(ptr)); }

// TwoSum(a.h, b.h) with the low parts added: a <- a + b.
__device__ __forceinline__ void df_add(DF2& a, const DF2& b) {
    float2 s = fadd2(a.h, b.h);
    float2 bb = fadd2(s, make_float2(-a.h.x, -a.h.y));
    float2 e1 = fadd2(a.h, make_float2(-(s.x - bb.x), -(s.y - bb.y)));
    float2 e2 = fadd2(b.h, make_float2(-bb.x, -bb.y));
    float2 e = fadd2(e1, e2);
    float2 l = fadd2(fadd2(a.l, b.l), e);
    a.h = s;
    a.l = l;
}

__device__ __forceinline__ float shfl_x(float x, int off) { return __shfl_xor_sync(0xffffffffu, x, off); }
__device__ __forceinline__ double shfl_x(double x, int off) { return __shfl_xor_sync(0xffffffffu, x, off); }

__device__ __forceinline__ float pow2f(int e) {   // 2^e as float for e in [-126, 127], 0 below
    return e < -126 ? 0.0f : __int_as_float((e + 127) << 23);
}

// Tile partial sum, before the Bloch phase and dV (k_tile_reduce applies both once per image segment).
// Layout [k*spin][tile slot (moff + m)][band], band fastest, so the reduce reads 32 bands of one slot in
// one coalesced access.  poff: offset of the table's slice (projections onto several tables), 0 otherwise.
__device__ __forceinline__ void write_partial(const View& v, const Tile& t, int ks, int band, int m, double re, double im,
                                              int64_t poff) {
    v.part[poff + ((int64_t)ks * v.TM + t.moff + m) * v.max_bands + band] = make_double2(re, im);
}

// Exact float -> double times 2^s with integer operations (the conversion instruction runs on the
// FP64 pipe).  Zeros and FP32 denormals give 0; s must keep the result normal.
__device__ __forceinline__ double f2d_scaled(float f, int s) {
    const unsigned u = __float_as_uint(f);
    const unsigned e = (u >> 23) & 0xFFu;
    const unsigned hi = (u & 0x80000000u) | ((e + 896u + (unsigned)s) << 20) | ((u & 0x7FFFFFu) >> 3);
    return e == 0 ? 0.0 : __hiloint2double((int)hi, (int)(u << 29));
}

// After the butterfly reductions every lane of a band's group holds the same sums, so the FP64
// epilogue (conversion, Bloch phase, dV) is spread over the lanes, one orbital each: it then issues
// once per warp instead of once per orbital on this GPU's narrow FP64 pipe.
template <int M, int Q, typename F>
__device__ __forceinline__ void per_lane_orbital(int q, F&& body) {
#pragma unroll
    for (int m0 = 0; m0 < M; m0 += Q)
        if (m0 + q < M) body(m0 + q);
}

// ------------------------------------------------------------------------------------------------
// F64 policy
// ------------------------------------------------------------------------------------------------
// x * (g.x + i g.y)
__device__ __forceinline__ double2 crot(double2 x, double2 g) {
    return make_double2(fma(g.x, x.x, -g.y * x.y), fma(g.y, x.x, g.x * x.y));
}

template <int M, int Q, int G>
__device__ __forceinline__ void proj_body_f64(const View& v, const Tile& t, int ks, int band, const double2* __restrict__ row,
                                              const int* s_idx, const double* s_phi, const double2* s_g, int64_t poff) {
    const int q = threadIdx.x & (Q - 1);
    double2 acc[M];
#pragma unroll
    for (int m = 0; m < M; ++m) acc[m] = make_double2(0.0, 0.0);
    if (row) {
        int i = q;
        for (; i + 3 * Q < t.np; i += 4 * Q) {
            double2 x[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) x[u] = __ldg(row + s_idx[i + u * Q]);
            if (G)
#pragma unroll
                for (int u = 0; u < 4; ++u) x[u] = crot(x[u], s_g[i + u * Q]);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const double* ph = s_phi + (i + u * Q) * M;
#pragma unroll
                for (int m = 0; m < M; ++m) {
                    acc[m].x = fma(ph[m], x[u].x, acc[m].x);
                    acc[m].y = fma(ph[m], x[u].y, acc[m].y);
                }
            }
        }
        for (; i < t.np; i += Q) {
            double2 x = __ldg(row + s_idx[i]);
            if (G) x = crot(x, s_g[i]);
            const double* ph = s_phi + i * M;
#pragma unroll
            for (int m = 0; m < M; ++m) {
                acc[m].x = fma(ph[m], x.x, acc[m].x);
                acc[m].y = fma(ph[m], x.y, acc[m].y);
            }
        }
    }
#pragma unroll
    for (int off = Q / 2; off > 0; off >>= 1)
#pragma unroll
        for (int m = 0; m < M; ++m) {
            acc[m].x += shfl_x(acc[m].x, off);
            acc[m].y += shfl_x(acc[m].y, off);
        }
    if (row)
        per_lane_orbital<M, Q>(q, [&](int mq) {
            double2 a = acc[0];
#pragma unroll
            for (int m = 1; m < M; ++m)
                if (m == mq) a = acc[m];
            write_partial(v, t, ks, band, mq, a.x, a.y, poff);
        });
}

// ------------------------------------------------------------------------------------------------
// F32 policy (complex64 states)
// ------------------------------------------------------------------------------------------------
// Orbital rows of a tile for this policy: per point 2*MP floats, [hi_0 .. hi_{MP-1}, lo_0 .. lo_{MP-1}]
// with MP = M rounded up to even (zero padding).  Products pair two orbitals against one broadcast
// state component, (phi_m, phi_m+1) x (x_re, x_re), so one 8-byte shared load feeds two orbitals:
// half the shared-memory wavefronts of a per-orbital (hi, hi, lo, lo) row, which bound this kernel.
template <int M, int Q, int CH, int PF, int G>
__device__ __forceinline__ void proj_body_f32(const View& v, const Tile& t, int ks, int band, const float2* __restrict__ row,
                                              const int* s_idx, const float* s_phf, const float4* s_g, int64_t poff) {
    constexpr int MP = (M + 1) & ~1, NP = MP / 2;
    const int q = threadIdx.x & (Q - 1);
    DF2 Rr[NP], Ri[NP];   // running sums of the real and imaginary parts of orbitals (2j, 2j+1)
#pragma unroll
    for (int j = 0; j < NP; ++j) {
        Rr[j] = DF2{make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
        Ri[j] = Rr[j];
    }
    if (row) {
        for (int i0 = q; i0 < t.np; i0 += Q * CH) {
            float2 x[CH];
#pragma unroll
            for (int c = 0; c < CH; ++c) {
                int i = i0 + c * Q;
                const bool in = i < t.np;
                x[c] = ld_gather(row + (in ? s_idx[i] : 0), in);
            }
            if (G)
#pragma unroll
                for (int c = 0; c < CH; ++c) {   // x * (cos + i sin) in FP32 (rows past the tile hold zeros)
                    const float4 g = s_g[i0 + c * Q];
                    x[c] = ffma2(make_float2(-g.y, g.x), make_float2(x[c].y, x[c].y),
                                 __fmul2_rn(make_float2(g.x, g.y), make_float2(x[c].x, x[c].x)));
                }
            if (PF) {
#pragma unroll
                for (int c = 0; c < CH; ++c) {
                    int i = i0 + Q * CH + c * Q;
                    if (i < t.np) prefetch_l2(row + s_idx[i]);
                }
            }
            DF2 cr[NP], ci[NP];
#pragma unroll
            for (int j = 0; j < NP; ++j) {
                cr[j] = DF2{make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
                ci[j] = cr[j];
            }
#pragma unroll
            for (int c = 0; c < CH; ++c) {
                const float* ph = s_phf + (i0 + c * Q) * (2 * MP);
                const float2 xr = make_float2(x[c].x, x[c].x), xi = make_float2(x[c].y, x[c].y);
#pragma unroll
                for (int j = 0; j < NP; ++j) {
                    const float2 h2 = *reinterpret_cast<const float2*>(ph + 2 * j);
                    const float2 l2 = *reinterpret_cast<const float2*>(ph + MP + 2 * j);
                    cr[j].h = ffma2(h2, xr, cr[j].h);
                    ci[j].h = ffma2(h2, xi, ci[j].h);
                    cr[j].l = ffma2(l2, xr, cr[j].l);
                    ci[j].l = ffma2(l2, xi, ci[j].l);
                }
            }
#pragma unroll
            for (int j = 0; j < NP; ++j) {
                df_add(Rr[j], cr[j]);
                df_add(Ri[j], ci[j]);
            }
        }
    }
#pragma unroll
    for (int off = Q / 2; off > 0; off >>= 1)
#pragma unroll
        for (int j = 0; j < NP; ++j) {
            DF2 o{make_float2(shfl_x(Rr[j].h.x, off), shfl_x(Rr[j].h.y, off)),
                  make_float2(shfl_x(Rr[j].l.x, off), shfl_x(Rr[j].l.y, off))};
            df_add(Rr[j], o);
            DF2 u{make_float2(shfl_x(Ri[j].h.x, off), shfl_x(Ri[j].h.y, off)),
                  make_float2(shfl_x(Ri[j].l.x, off), shfl_x(Ri[j].l.y, off))};
            df_add(Ri[j], u);
        }
    if (row)
        per_lane_orbital<M, Q>(q, [&](int mq) {
            float rh = Rr[0].h.x, rl = Rr[0].l.x, ih = Ri[0].h.x, il = Ri[0].l.x;
#pragma unroll
            for (int m = 1; m < M; ++m)
                if (m == mq) {
                    const DF2& a = Rr[m / 2];
                    const DF2& b = Ri[m / 2];
                    rh = (m & 1) ? a.h.y : a.h.x;
                    rl = (m & 1) ? a.l.y : a.l.x;
                    ih = (m & 1) ? b.h.y : b.h.x;
                    il = (m & 1) ? b.l.y : b.l.x;
                }
            write_partial(v, t, ks, band, mq, f2d_scaled(rh, 0) + f2d_scaled(rl, 0), f2d_scaled(ih, 0) + f2d_scaled(il, 0), poff);
        });
}

// ------------------------------------------------------------------------------------------------
// PAIR policy (complex128 states, FP32-pair arithmetic)
// ------------------------------------------------------------------------------------------------
// Split a double x with biased exponent field E <= Em (Em >= 127, the chain's largest) into floats
// hi + lo of x * 2^(1023-Em) by assembling their bit patterns with integer operations: hi takes the
// sign, the exponent E - Em + 127 and the top 23 fraction bits (a funnel shift of the two words after
// the exponent is rebased in place); lo the next 23 fraction bits under the exponent of hi less 23,
// minus the implicit one of that pattern (an exact subtraction).  47 significant bits, error below
// 2^-46 of 2^(E-Em).  bias = (Em - 127) << 20.  Magnitudes more than 2^103 below 2^(Em-1023), zeros
// included, are raised to that floor (an absolute change below 2^-102 of the chain scale), so both
// exponents stay normal without a branch.
__device__ __forceinline__ void split_bits(double x, int bias, float& hi, float& lo) {
    const unsigned whi = (unsigned)__double2hiint(x), wlo = (unsigned)__double2loint(x);
    const int a = max((int)(whi & 0x7FFFFFFFu) - bias, 24 << 20);                 // exponent field E' >= 24
    const unsigned hb = __funnelshift_l(wlo, (unsigned)a, 3) | (whi & 0x80000000u);
    const unsigned one = (hb - (23u << 23)) & 0xFF800000u;                         // +-2^(E' - 150)
    hi = __uint_as_float(hb);
    lo = __uint_as_float(one | ((wlo >> 6) & 0x007FFFFFu)) - __uint_as_float(one);
}

// the exponent field of x in place (a mask other than the split's, so the compiler does not keep one
// shared masked word per point alive across the chain)
__device__ __forceinline__ unsigned exp_bits(double x) { return (unsigned)__double2hiint(x) & 0x7FF00000u; }

// (bh + bl) * (g.x + g.z + i (g.y + g.w)) as a new float pair, componentwise for (re, im): the hi
// products are formed exactly (product + FMA residual) and added with TwoSum, the cross terms with
// the low parts go into the low word.  Error ~2^-47 of |b|; the modulus grows by at most sqrt(2) per
// component.
__device__ __forceinline__ void rot_pair(float2& bh, float2& bl, float4 g) {
    const float2 uh = make_float2(g.x, g.y), wh = make_float2(-g.y, g.x);
    const float2 ul = make_float2(g.z, g.w), wl = make_float2(-g.w, g.z);
    const float2 xr = make_float2(bh.x, bh.x), xi = make_float2(bh.y, bh.y);
    const float2 P = __fmul2_rn(uh, xr), R = __fmul2_rn(wh, xi);
    const float2 eP = ffma2(uh, xr, make_float2(-P.x, -P.y));
    const float2 eR = ffma2(wh, xi, make_float2(-R.x, -R.y));
    const float2 s = fadd2(P, R);
    const float2 bb = fadd2(s, make_float2(-P.x, -P.y));
    const float2 t = fadd2(fadd2(P, make_float2(bb.x - s.x, bb.y - s.y)), fadd2(R, make_float2(-bb.x, -bb.y)));
    float2 lo = fadd2(fadd2(eP, eR), t);
    lo = ffma2(uh, make_float2(bl.x, bl.x), lo);
    lo = ffma2(ul, xr, lo);
    lo = ffma2(wh, make_float2(bl.y, bl.y), lo);
    lo = ffma2(wl, xi, lo);
    bh = s;
    bl = lo;
}

// The Q*CH-point chain starting at i0 (lane points i0 + c*Q) into registers, zeros past the tile.
template <int Q, int CH>
__device__ __forceinline__ void pair_load(double2 (&x)[CH], int i0, const double2* __restrict__ row, const int* s_idx, int np) {
#pragma unroll
    for (int c = 0; c < CH; ++c) {
        int i = i0 + c * Q;
        x[c] = (i < np) ? __ldg(row + s_idx[i]) : make_double2(0.0, 0.0);
    }
}

// One chain of the FP32-pair projection: the chain's scale (Em_run rises to its largest exponent and R
// is rescaled), the split states, the offset-accumulated products, merged into R.
template <int M, int Q, int CH, int G>
__device__ __forceinline__ void pair_chain(const double2 (&x)[CH], int i0, DF2 (&R)[M], int& Em_run, bool& bad, float Cv,
                                           const float4* s_phi, const float4* s_g) {
    const float2 C2 = make_float2(Cv, Cv);
    const float2 mone = make_float2(-1.f, -1.f);
    unsigned am = 0;
#pragma unroll
    for (int c = 0; c < CH; ++c) am = max(am, max(exp_bits(x[c].x), exp_bits(x[c].y)));
    int Ec = (int)(am >> 20);
    if (Ec == 0x7FF) bad = true;
    if (Ec == 0) return;
    Ec = max(Ec, 127);   // the split needs Em >= 127 (zeros then scale to 0)
    if (Ec > Em_run) {
        if (Em_run != 0) {
            float s = pow2f(Em_run - Ec);
            float2 s2 = make_float2(s, s);
#pragma unroll
            for (int m = 0; m < M; ++m) {
                R[m].h = __fmul2_rn(R[m].h, s2);
                R[m].l = __fmul2_rn(R[m].l, s2);
            }
        }
        Em_run = Ec;
    }
    float2 acc[M], lo[M];
#pragma unroll
    for (int m = 0; m < M; ++m) { acc[m] = C2; lo[m] = make_float2(0.f, 0.f); }
    const int bias = (Em_run - 127) << 20;
#pragma unroll
    for (int c = 0; c < CH; ++c) {
        float2 bh, bl;
        split_bits(x[c].x, bias, bh.x, bl.x);
        split_bits(x[c].y, bias, bh.y, bl.y);
        if (G) rot_pair(bh, bl, s_g[i0 + c * Q]);
        const float4* ph = s_phi + (i0 + c * Q) * M;
#pragma unroll
        for (int m = 0; m < M; ++m) {
            float4 f = ph[m];                                  // (hi, hi, lo, lo)
            float2 ah = make_float2(f.x, f.y), al = make_float2(f.z, f.w);
            float2 s = ffma2(ah, bh, acc[m]);                  // acc + a*b, rounded
            float2 tneg = ffma2(s, mone, acc[m]);              // acc - s  (exact: same binade)
            float2 r = ffma2(ah, bh, tneg);                    // rounding residual a*b - (s - acc)
            lo[m] = fadd2(lo[m], r);
            lo[m] = ffma2(ah, bl, lo[m]);
            lo[m] = ffma2(al, bh, lo[m]);
            acc[m] = s;
        }
    }
#pragma unroll
    for (int m = 0; m < M; ++m) {
        DF2 chn{fadd2(acc[m], make_float2(-Cv, -Cv)), lo[m]};  // exact removal of the offset
        df_add(R[m], chn);
    }
}

// Each lane takes chains of CH points (i0 + c*Q), one after another, and merges each into R.
// PF = 1: every chain asks L2 for the next one; PF = 5: in addition the last chain of the tile asks for
// the first chain of the band the lane takes next (row_next, null if none), so only the first band
// group of a CTA starts cold.
template <int M, int Q, int CH, int PF, int G>
__device__ __forceinline__ void proj_body_pair(const View& v, const Tile& t, int ks, int band, const double2* __restrict__ row,
                                               const double2* __restrict__ row_next, const int* s_idx, const float4* s_phi,
                                               int pe, const float4* s_g, int64_t poff) {
    const int q = threadIdx.x & (Q - 1);
    DF2 R[M];
#pragma unroll
    for (int m = 0; m < M; ++m) R[m] = DF2{make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
    int Em_run = 0;
    bool bad = false;
    // chain offset C = 2^(pe + 1 + log2 CH + 2) >= 4 * CH * max|phi x'|, |x'| < 2, |phi| < 2^pe
    // (one more power of two when x' is rotated by a gauge phase: |x'| < 2 sqrt 2)
    constexpr int LOG2CH = (CH >= 16) ? 4 : (CH >= 8) ? 3 : (CH >= 4) ? 2 : (CH >= 2) ? 1 : 0;
    const float Cv = pow2f(min(max(pe + 3 + G + LOG2CH, -100), 100));
#define DFTU_PAIR_CHAIN(x, i0) pair_chain<M, Q, CH, G>(x, i0, R, Em_run, bad, Cv, s_phi, s_g)
#define DFTU_PAIR_LOAD(x, i0) pair_load<Q, CH>(x, i0, row, s_idx, t.np)
    // L2 prefetch of the chain starting at i0; past the tile (PF == 5) the first chain of the next band
    auto prefetch = [&](int i0) {
        if (PF == 1 || PF == 5 || (PF == 2 && (q == 0 || q == Q - 1))) {   // PF == 2: the group's edge lanes only
            if (PF == 5 && i0 >= t.np) {
                if (row_next)
#pragma unroll
                    for (int c = 0; c < CH; ++c) {
                        int i = q + c * Q;
                        if (i < t.np) prefetch_l2(row_next + s_idx[i]);
                    }
            } else {
#pragma unroll
                for (int c = 0; c < CH; ++c) {
                    int i = i0 + c * Q;
                    if (i < t.np) prefetch_l2(row + s_idx[i]);
                }
            }
        }
    };
    if (row)
        for (int i0 = q; i0 < t.np; i0 += Q * CH) {
            double2 x[CH];
            DFTU_PAIR_LOAD(x, i0);
            prefetch(i0 + Q * CH);
            DFTU_PAIR_CHAIN(x, i0);
        }
#undef DFTU_PAIR_CHAIN
#undef DFTU_PAIR_LOAD
    // bring the Q lanes of this band to a common scale, then add in pairs
    int Em_max = Em_run;
#pragma unroll
    for (int off = Q / 2; off > 0; off >>= 1) Em_max = max(Em_max, __shfl_xor_sync(0xffffffffu, Em_max, off));
    if (Em_run != Em_max) {
        float s = (Em_run == 0) ? 0.0f : pow2f(Em_run - Em_max);
        float2 s2 = make_float2(s, s);
#pragma unroll
        for (int m = 0; m < M; ++m) {
            R[m].h = __fmul2_rn(R[m].h, s2);
            R[m].l = __fmul2_rn(R[m].l, s2);
        }
    }
#pragma unroll
    for (int off = Q / 2; off > 0; off >>= 1)
#pragma unroll
        for (int m = 0; m < M; ++m) {
            DF2 o{make_float2(shfl_x(R[m].h.x, off), shfl_x(R[m].h.y, off)),
                  make_float2(shfl_x(R[m].l.x, off), shfl_x(R[m].l.y, off))};
            df_add(R[m], o);
        }
    int anybad = bad ? 1 : 0;   // any non-finite value among this band's lanes
#pragma unroll
    for (int off = Q / 2; off > 0; off >>= 1) anybad |= __shfl_xor_sync(0xffffffffu, anybad, off);
    if (row) {
        const int sc = Em_max - 1023;   // the sums are in units of 2^(Em_max - 1023), Em_max >= 127 or sums zero
        per_lane_orbital<M, Q>(q, [&](int mq) {
            DF2 a = R[0];
#pragma unroll
            for (int m = 1; m < M; ++m)
                if (m == mq) a = R[m];
            double re = f2d_scaled(a.h.x, sc) + f2d_scaled(a.l.x, sc);
            double im = f2d_scaled(a.h.y, sc) + f2d_scaled(a.l.y, sc);
            if (anybad) { re = __longlong_as_double(0x7FF8000000000000LL); im = re; }
            write_partial(v, t, ks, band, mq, re, im, poff);
        });
    }
}

// ------------------------------------------------------------------------------------------------
// F32 policy, two bands per lane (complex64 states)
// ------------------------------------------------------------------------------------------------
// Every lane walks its points for two bands at once, so each grid index and each paired orbital load
// from shared memory serves both.  Products are compensated as in proj_body_f32 (phi = hi + lo, both
// halves multiplied by the FP32 state value); the sums are plain FP32 over the lane's points of the
// tile, then over the Q lanes, and FP64 from there on (across tiles).
// FOLD: each product phi x is formed from both halves of phi by two fused multiply-adds into one FP32 sum
// (hi then lo), instead of separate sums of the hi and lo products: half the accumulator registers, the
// same products; the lo half then enters at the sum's rounding, which plain FP32 accumulation over a
// lane's points already sets.
template <int M, int Q, int CH, int PF, int FOLD = 0>
__device__ __forceinline__ void proj_body_f32x2(const View& v, const Tile& t, int ks, int band, int nbands,
                                                const float2* __restrict__ row0, const float2* __restrict__ row1,
                                                const int* s_idx, const float* s_phf, int64_t poff) {
    constexpr int MP = (M + 1) & ~1, NP = MP / 2;
    constexpr int NS = FOLD ? 2 : 4;
    const int q = threadIdx.x & (Q - 1);
    // [band][part]: real hi, imaginary hi (real lo, imaginary lo unless folded) of orbitals (2j, 2j+1)
    float2 S0[NS][NP], S1[NS][NP];
#pragma unroll
    for (int a = 0; a < NS; ++a)
#pragma unroll
        for (int j = 0; j < NP; ++j) { S0[a][j] = make_float2(0.f, 0.f); S1[a][j] = S0[a][j]; }
    if (row0) {
        for (int i0 = q; i0 < t.np; i0 += Q * CH) {
            float2 x0[CH], x1[CH];
#pragma unroll
            for (int c = 0; c < CH; ++c) {
                const int i = i0 + c * Q;
                const bool in = i < t.np;
                const int g = in ? s_idx[i] : 0;
                x0[c] = ld_gather(row0 + g, in);
                x1[c] = ld_gather(row1 + g, in && row1);
            }
            if (PF) {
                // PF == 2: only the first and last lane of a band's group, whose points bound the Q
                // consecutive points the group reads next (at most two 128-byte lines per row)
                if (PF == 1 || q == 0 || q == Q - 1) {
#pragma unroll
                    for (int c = 0; c < CH; ++c) {
                        const int i = i0 + Q * CH + c * Q;
                        if (i < t.np) {
                            prefetch_l2(row0 + s_idx[i]);
                            if (row1) prefetch_l2(row1 + s_idx[i]);
                        }
                    }
                }
            }
#pragma unroll
            for (int c = 0; c < CH; ++c) {
                const float* ph = s_phf + (i0 + c * Q) * (2 * MP);
                const float2 r0 = make_float2(x0[c].x, x0[c].x), m0 = make_float2(x0[c].y, x0[c].y);
                const float2 r1 = make_float2(x1[c].x, x1[c].x), m1 = make_float2(x1[c].y, x1[c].y);
#pragma unroll
                for (int j = 0; j < NP; ++j) {
                    const float2 h2 = *reinterpret_cast<const float2*>(ph + 2 * j);
                    const float2 l2 = *reinterpret_cast<const float2*>(ph + MP + 2 * j);
                    if (FOLD) {
                        S0[0][j] = ffma2(l2, r0, ffma2(h2, r0, S0[0][j]));
                        S0[1][j] = ffma2(l2, m0, ffma2(h2, m0, S0[1][j]));
                        S1[0][j] = ffma2(l2, r1, ffma2(h2, r1, S1[0][j]));
                        S1[1][j] = ffma2(l2, m1, ffma2(h2, m1, S1[1][j]));
                    } else {
                        S0[0][j] = ffma2(h2, r0, S0[0][j]); S0[1][j] = ffma2(h2, m0, S0[1][j]);
                        S0[NS - 2][j] = ffma2(l2, r0, S0[NS - 2][j]); S0[NS - 1][j] = ffma2(l2, m0, S0[NS - 1][j]);
                        S1[0][j] = ffma2(h2, r1, S1[0][j]); S1[1][j] = ffma2(h2, m1, S1[1][j]);
                        S1[NS - 2][j] = ffma2(l2, r1, S1[NS - 2][j]); S1[NS - 1][j] = ffma2(l2, m1, S1[NS - 1][j]);
                    }
                }
            }
        }
    }
#pragma unroll
    for (int off = Q / 2; off > 0; off >>= 1)
#pragma unroll
        for (int a = 0; a < NS; ++a)
#pragma unroll
            for (int j = 0; j < NP; ++j) {
                S0[a][j] = fadd2(S0[a][j], make_float2(shfl_x(S0[a][j].x, off), shfl_x(S0[a][j].y, off)));
                S1[a][j] = fadd2(S1[a][j], make_float2(shfl_x(S1[a][j].x, off), shfl_x(S1[a][j].y, off)));
            }
    if (row0) {
        per_lane_orbital<M, Q>(q, [&](int mq) {
#pragma unroll
            for (int b = 0; b < 2; ++b) {
                if (b == 1 && !row1) break;
                float v4[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                for (int a = 0; a < NS; ++a) {
                    const float2 w = (b == 0) ? S0[a][0] : S1[a][0];
                    v4[a] = w.x;
                }
#pragma unroll
                for (int m = 1; m < M; ++m)
                    if (m == mq)
#pragma unroll
                        for (int a = 0; a < NS; ++a) {
                            const float2 w = (b == 0) ? S0[a][m / 2] : S1[a][m / 2];
                            v4[a] = (m & 1) ? w.y : w.x;
                        }
                write_partial(v, t, ks, band + b, mq, f2d_scaled(v4[0], 0) + f2d_scaled(v4[2], 0),
                              f2d_scaled(v4[1], 0) + f2d_scaled(v4[3], 0), poff);
            }
        });
    }
    (void)nbands;
}

// ------------------------------------------------------------------------------------------------
// kernels
// ------------------------------------------------------------------------------------------------
enum Pol { P_F64 = 0, P_PAIR = 1, P_F32 = 2, P_F32B2 = 4, P_F32B2F = 5 };

// bands a lane carries at once
template <int POL> struct LaneBands { static constexpr int value = (POL == P_F32B2 || POL == P_F32B2F) ? 2 : 1; };

// Bytes of one staged orbital row (one point) for the largest shell maxM: FP64 values, (hi, hi, lo, lo)
// per orbital for the FP32-pair policy, [hi pairs | lo pairs] for the complex64 policies.
__host__ __device__ constexpr size_t phi_row_bytes(int pol, int maxM) {
    return pol == P_F64 ? 8 * (size_t)maxM : pol == P_PAIR ? 16 * (size_t)maxM : 8 * (size_t)((maxM + 1) & ~1);
}

// The bands of one group, [band0, band0 + NT/Q * bands per lane), over the staged tile.  more: a full group of the
// same shape follows.  HOIST: what comes from outside the loop over groups (1: k and s, 2: the orbitals' exponent); the
// kernels sit at the register limit of their occupancy, and each form keeps its registers one way only (2048 oxide
// states: eight groups fixed 2079 us with 1 against 2113, complex64 with 0 1093 against 1112).
template <int POL, int Q, int CH, int PF, int G, int NT, int TP, int HOIST>
__device__ __forceinline__ void project_group(const View& v, const Tile& t, const ProjArgs& a, int ks, int k0, int s0, int band0, bool more, const int* s_pe, int pe0,
                                              const unsigned char* smem, const unsigned char* s_gauge, int64_t poff) {
    const int* s_idx = reinterpret_cast<const int*>(smem);
    constexpr int NBL = LaneBands<POL>::value;   // bands per lane
    constexpr int BPW = (32 / Q) * NBL;
    constexpr int BPC = (NT / 32) * BPW;
    const int k = HOIST == 1 ? k0 : ks / v.ns, s = HOIST == 1 ? s0 : ks % v.ns;
    const int band = band0 + (threadIdx.x >> 5) * BPW + ((threadIdx.x & 31) / Q) * NBL;
    const bool active = band < a.nbands;
    const int64_t off = (int64_t)k * a.sk + (int64_t)s * a.ss + (int64_t)band * a.sn;
    if (POL == P_F32B2 || POL == P_F32B2F) {
        constexpr int FOLD = (POL == P_F32B2F) ? 1 : 0;
        const float* s_phf = reinterpret_cast<const float*>(smem + TP * sizeof(int));
        const float2* row0 = active ? reinterpret_cast<const float2*>(a.psi) + off : nullptr;
        const float2* row1 = (band + 1 < a.nbands) ? row0 + a.sn : nullptr;
        switch (t.M) {
            case 1: proj_body_f32x2<1, Q, CH, PF, FOLD>(v, t, ks, band, a.nbands, row0, row1, s_idx, s_phf, poff); break;
            case 3: proj_body_f32x2<3, Q, CH, PF, FOLD>(v, t, ks, band, a.nbands, row0, row1, s_idx, s_phf, poff); break;
            case 5: proj_body_f32x2<5, Q, CH, PF, FOLD>(v, t, ks, band, a.nbands, row0, row1, s_idx, s_phf, poff); break;
            // an f shell's sums leave registers for half the loads in flight (the order of its sums is the same)
            default: proj_body_f32x2<7, Q, FOLD ? CH / 2 : CH, PF, FOLD>(v, t, ks, band, a.nbands, row0, row1, s_idx, s_phf, poff); break;
        }
    } else if (POL == P_F64) {
        const double* s_phi = reinterpret_cast<const double*>(smem + TP * sizeof(int));
        const double2* row = active ? reinterpret_cast<const double2*>(a.psi) + off : nullptr;
        const double2* s_g = reinterpret_cast<const double2*>(s_gauge);
        switch (t.M) {
            case 1: proj_body_f64<1, Q, G>(v, t, ks, band, row, s_idx, s_phi, s_g, poff); break;
            case 3: proj_body_f64<3, Q, G>(v, t, ks, band, row, s_idx, s_phi, s_g, poff); break;
            case 5: proj_body_f64<5, Q, G>(v, t, ks, band, row, s_idx, s_phi, s_g, poff); break;
            default: proj_body_f64<7, Q, G>(v, t, ks, band, row, s_idx, s_phi, s_g, poff); break;
        }
    } else if (POL == P_PAIR) {
        const float4* s_phi = reinterpret_cast<const float4*>(smem + TP * sizeof(int));
        const double2* row = active ? reinterpret_cast<const double2*>(a.psi) + off : nullptr;
        const double2* row_next = (active && more && band + BPC < a.nbands) ? row + (int64_t)BPC * a.sn : nullptr;
        const int pe = HOIST == 2 ? pe0 : *s_pe;
        const float4* s_g = reinterpret_cast<const float4*>(s_gauge);
        switch (t.M) {
            case 1: proj_body_pair<1, Q, CH, PF, G>(v, t, ks, band, row, row_next, s_idx, s_phi, pe, s_g, poff); break;
            case 3: proj_body_pair<3, Q, CH, PF, G>(v, t, ks, band, row, row_next, s_idx, s_phi, pe, s_g, poff); break;
            case 5: proj_body_pair<5, Q, CH, PF, G>(v, t, ks, band, row, row_next, s_idx, s_phi, pe, s_g, poff); break;
            default: proj_body_pair<7, Q, CH, PF, G>(v, t, ks, band, row, row_next, s_idx, s_phi, pe, s_g, poff); break;
        }
    } else {
        const float* s_phf = reinterpret_cast<const float*>(smem + TP * sizeof(int));
        const float2* row = active ? reinterpret_cast<const float2*>(a.psi) + off : nullptr;
        const float4* s_g = reinterpret_cast<const float4*>(s_gauge);
        switch (t.M) {
            case 1: proj_body_f32<1, Q, CH, PF, G>(v, t, ks, band, row, s_idx, s_phf, s_g, poff); break;
            case 3: proj_body_f32<3, Q, CH, PF, G>(v, t, ks, band, row, s_idx, s_phf, s_g, poff); break;
            case 5: proj_body_f32<5, Q, CH, PF, G>(v, t, ks, band, row, s_idx, s_phf, s_g, poff); break;
            default: proj_body_f32<7, Q, CH, PF, G>(v, t, ks, band, row, s_idx, s_phf, s_g, poff); break;
        }
    }
}

// One work item: tile `tile_id` of the system described by (v, a), spin/component index ks, every band of
// band chunk `chunk` (NBG groups of BPC bands, nbg when NBG is 0), against orbital table `dir` (0 unless the launch projects
// onto several tables).  The tile is staged in shared memory once.  TP: the tiling's largest tile (TILE,
// or PTILE when the launch's View carries the projection's own tiling); shared memory holds TP grid
// indices, then TP + 128 orbital rows (zeros past the tile), then the gauge phases.
template <int POL, int Q, int CH, int NBG, int PF, int G, int NT = CTA, int TP = TILE, int TAIL = 0>
__device__ __forceinline__ void project_item(const View& v, const ProjArgs& a, int tile_id, int ks, int chunk, int nbg,
                                             unsigned char* smem, int* s_pe, int dir = 0) {
    int* s_idx = reinterpret_cast<int*>(smem);
    if (G) dependent_wait();   // the phase table may be the kernel before's
    const Tile t = v.tiles[tile_id];
    const int k = ks / v.ns, s = ks % v.ns;
    const int64_t ph0 = t.phi0 + dir * v.phi_dir_stride;   // this table's rows of the tile
    const int64_t poff = dir * v.part_dir_stride;
    constexpr int NBL = LaneBands<POL>::value;   // bands per lane
    constexpr int BPW = (32 / Q) * NBL;
    constexpr int BPC = (NT / 32) * BPW;

    // ---- stage the tile once (grid indices, orbital rows, orbital exponent bound)
    if (threadIdx.x == 0) *s_pe = -200;
    constexpr int TPAD = TP + (TILE_PAD - TILE);
    for (int i = threadIdx.x; i < TP; i += NT) s_idx[i] = (i < t.np) ? v.pt_idx[t.p0 + i] : 0;
    __syncthreads();
    if (POL == P_F64) {
        double* s_phi = reinterpret_cast<double*>(smem + TP * sizeof(int));
        for (int e = threadIdx.x; e < TP * t.M; e += NT)
            s_phi[e] = (e < t.np * t.M) ? v.phi64[ph0 + e] : 0.0;
    } else if (POL == P_F32 || POL == P_F32B2 || POL == P_F32B2F) {
        float* s_phf = reinterpret_cast<float*>(smem + TP * sizeof(int));
        const int MP = (t.M + 1) & ~1;
        int pe = -200;
        for (int e = threadIdx.x; e < TPAD * MP; e += NT) {
            const int i = e / MP, m = e - i * MP;
            float hi = 0.f, lo = 0.f;
            if (i < t.np && m < t.M) { hi = v.phi_hi[ph0 + (int64_t)i * t.M + m]; lo = v.phi_lo[ph0 + (int64_t)i * t.M + m]; }
            s_phf[i * 2 * MP + m] = hi;
            s_phf[i * 2 * MP + MP + m] = lo;
            if (hi != 0.f) pe = max(pe, ((__float_as_int(hi) >> 23) & 0xFF) - 127 + 1);   // |hi| < 2^pe
        }
    } else {
        float4* s_phi = reinterpret_cast<float4*>(smem + TP * sizeof(int));
        int pe = -200;
        for (int e = threadIdx.x; e < TPAD * t.M; e += NT) {
            float hi = 0.f, lo = 0.f;
            if (e < t.np * t.M) { hi = v.phi_hi[ph0 + e]; lo = v.phi_lo[ph0 + e]; }
            s_phi[e] = make_float4(hi, hi, lo, lo);
            if (hi != 0.f) pe = max(pe, ((__float_as_int(hi) >> 23) & 0xFF) - 127 + 1);   // |hi| < 2^pe
        }
        if (POL == P_PAIR) atomicMax(s_pe, pe);
    }
    // gauge phases of the tile's points (zeros past the tile), after the orbital rows of the largest shell
    unsigned char* s_gauge = smem + TP * sizeof(int) + (size_t)TPAD * phi_row_bytes(POL, v.maxM);
    if (G) {
        if (POL == P_F64)
            for (int i = threadIdx.x; i < TPAD; i += NT)
                reinterpret_cast<double2*>(s_gauge)[i] = (i < t.np) ? v.gauge_d[t.p0 + i] : make_double2(0.0, 0.0);
        else
            for (int i = threadIdx.x; i < TPAD; i += NT)
                reinterpret_cast<float4*>(s_gauge)[i] = (i < t.np) ? v.gauge_f[t.p0 + i] : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    __syncthreads();

    // ---- stream nbg groups of BPC bands over the staged tile
    // TAIL: a last group with few bands takes more lanes per band: its chains get shorter instead of warps idling
    // (65 complex128 bands are two groups of 32 and one of one band, which used to cost as much as a full one).
    dependent_wait();   // the states
    constexpr int HOIST = POL != P_PAIR ? 0 : !TAIL ? (NBG != 0) : NBG == 0 ? 2 : 0;
    const int pe = HOIST == 2 ? *s_pe : 0;
    const int ng = NBG ? NBG : nbg;
    for (int g = 0; g < ng; ++g) {
        const int band0 = (chunk * ng + g) * BPC;
        if (band0 >= a.nbands) break;
        const int left = a.nbands - band0;
        if (TAIL && left <= BPC / 4) project_group<POL, TAIL ? 32 : Q, TAIL ? 4 : CH, 0, G, NT, TP, HOIST>(v, t, a, ks, k, s, band0, false, s_pe, pe, smem, s_gauge, poff);
        else if (TAIL && left <= BPC / 2) project_group<POL, TAIL ? 16 : Q, TAIL ? 8 : CH, 0, G, NT, TP, HOIST>(v, t, a, ks, k, s, band0, false, s_pe, pe, smem, s_gauge, poff);
        else project_group<POL, Q, CH, PF, G, NT, TP, HOIST>(v, t, a, ks, k, s, band0, g + 1 < ng, s_pe, pe, smem, s_gauge, poff);
    }
}

// NDIR > 1: blockIdx.x = tile * NDIR + table, so the CTAs of one tile and band chunk for the
// NDIR orbital tables are neighbours in the launch and read the same states while they sit in L2.
template <int POL, int Q, int CH, int NBG, int PF, int MINB, int G, int NDIR = 1, int NT = CTA, int TP = TILE, int TAIL = 0>
__global__ void __launch_bounds__(NT, MINB) k_project(View v, ProjArgs a, int nbg) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int s_pe;
    const int tile = (NDIR == 1) ? (int)blockIdx.x : (int)blockIdx.x / NDIR;
    const int dir = (NDIR == 1) ? 0 : (int)blockIdx.x % NDIR;
    if (NDIR > 1 && dir >= cur_tables(v.tiles[tile].M)) return;   // the atom has fewer tables
    project_item<POL, Q, CH, NBG, PF, G, NT, TP, TAIL>(v, a, tile, blockIdx.z, blockIdx.y, nbg, smem, &s_pe, dir);
}

// Persistent form over many systems: every CTA takes (system, tile, k*spin) items from a counter until
// the list is exhausted and processes all band chunks of the item's system.
template <int POL, int Q, int CH, int NBG, int PF, int MINB, int NT = CTA>
__global__ void __launch_bounds__(NT, MINB) k_project_batch(const View* __restrict__ views, const ProjArgs* __restrict__ args,
                                                          const int4* __restrict__ items, int nitems, int* counter) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int s_pe, s_item;
    constexpr int BPC = (NT / 32) * (32 / Q) * LaneBands<POL>::value;
    for (;;) {
        if (threadIdx.x == 0) s_item = atomicAdd(counter, 1);
        __syncthreads();
        const int it = s_item;
        if (it >= nitems) break;
        const int4 w = items[it];   // (system, tile, k*spin, unused)
        const View& v = views[w.x];
        const ProjArgs& a = args[w.x];
        const int nchunks = (a.nbands + BPC * NBG - 1) / (BPC * NBG);
        for (int c = 0; c < nchunks; ++c) {
            project_item<POL, Q, CH, NBG, PF, 0, NT>(v, a, w.y, w.z, c, NBG, smem, &s_pe);
            __syncthreads();   // the next chunk or item restages shared memory
        }
    }
}

// Whether MINB CTAs of fn with smem bytes of dynamic shared memory fit on one SM (cached per kernel and size).
bool fits_per_sm(const void* fn, int nt, size_t smem, int minb);

// Bands groups per CTA, at most `most`: the count with the least waves x (staging + groups) of the grid, staging a
// tile counted as 0.35 of a group (a 1024-point tile: 96 KB into shared memory against 512 KB of states).  Large
// grids keep `most`; where a wave would be mostly empty, fewer groups fill it.
inline int balanced_groups(int most, int bands_per_group, int nbands, int64_t tiles, int64_t slots) {
    const int groups = (nbands + bands_per_group - 1) / bands_per_group;
    int best = most;
    double least = 1e300;
    for (int g = std::min(most, groups); g >= 1; --g) {
        const int64_t ctas = tiles * ((groups + g - 1) / g);
        // beyond a few waves the SMs share the work out whatever the split: every CTA's staging and every group once
        const double cost = ctas >= 4 * slots ? (ctas * 0.35 + (double)tiles * groups) / slots : (double)((ctas + slots - 1) / slots) * (0.35 + g);
        if (cost < 0.97 * least) { least = cost; best = g; }
    }
    return best;
}

// One projection launch.  TP = PTILE runs over the projection's own tiling (View::ptiles) when MINB CTAs
// with that shared memory still fit on an SM, and over the TILE tiling otherwise; *used receives the View
// the launch ran with, whose tiling the tile reduce must follow.
// BAL: the band groups per CTA follow the grid, up to NBG (at run time for the FP32-pair kernel; the complex64 kernel
// spills with a run-time count and is compiled for NBG, NBG / 2 and 1).
// RAGGED: a last group at most half full may take the kernel in which such groups have more lanes per band.  The
// three forms are kernels of their own, because the others' code costs the full groups registers that spill: 2048 oxide
// states take 2079 us with eight groups fixed, 2111 with the count at run time and ragged groups in the kernel.  So
// - eight groups fixed where that is the split (232 bands, four k: 1932 us against 1951 with the ragged form);
// - with a balanced split below that, the ragged form (40, 72 and 136 bands: 423, 681 and 1185 us against 461, 704 and
//   1205; half full groups are equal);
// - under a vector potential and for the current, eight groups fixed at any size, the ragged form where the last group
//   counts for much (40, 65 and 264 bands: 527, 788 and 2859 against 562, 821 and 2939; 80 and 112 bands would take
//   944 and 1284 against 933 and 1262).
template <int POL, int Q, int CH, int NBG, int PF, int MINB = 2, int G = 0, int NDIR = 1, int NT = CTA, int TP = TILE, bool BAL = false,
          bool RAGGED = false>
static cudaError_t run_project(const View& v, const ProjArgs& a, cudaStream_t st, View* used = nullptr) {
    static_assert(Q * CH <= TILE_PAD - TILE, "chained loops read up to Q*CH rows past the tile");
    static_assert(TP == TILE || TP == PTILE, "a tiling the View carries");
    static_assert(!RAGGED || (POL == P_PAIR && Q == 8 && CH == 8), "the ragged groups' shapes");
    constexpr int TPAD = TP + (TILE_PAD - TILE);
    size_t smem = TP * sizeof(int) + (size_t)TPAD * phi_row_bytes(POL, v.maxM) + (G ? (size_t)TPAD * 16 : 0);
    auto fn = k_project<POL, Q, CH, NBG, PF, MINB, G, NDIR, NT, TP>;
    View vl = v;
    if (TP != TILE) {
        if (!fits_per_sm((const void*)fn, NT, smem, MINB)) return run_project<POL, Q, CH, NBG, PF, MINB, G, NDIR, NT, TILE, BAL, RAGGED>(v, a, st, used);
        vl.tiles = v.ptiles; vl.ntiles = v.nptiles; vl.TM = v.pTM;
        vl.atom_tile_beg = v.patom_tile_beg; vl.atom_tile_end = v.patom_tile_end;
    }
    if (used) *used = vl;
    constexpr int BPC = (NT / 32) * (32 / Q) * LaneBands<POL>::value;
    const int nbg = BAL ? balanced_groups(NBG, BPC, a.nbands, (int64_t)vl.ntiles * NDIR * vl.nk * vl.ns, MINB * sm_count()) : NBG;
    if constexpr (BAL && POL == P_PAIR)
        if (nbg != NBG) fn = k_project<POL, Q, CH, 0, PF, MINB, G, NDIR, NT, TP>;
    if constexpr (RAGGED) {
        const int left = a.nbands % BPC, groups = (a.nbands + BPC - 1) / BPC;
        const bool pays = BAL ? nbg != NBG : NBG == 1 || groups == 1 || (left <= BPC / 4 && (groups <= 3 || groups % NBG == 1));
        if (left > 0 && left <= BPC / 2 && pays) fn = k_project<POL, Q, CH, BAL ? 0 : NBG, PF, MINB, G, NDIR, NT, TP, 1>;
    }
    cudaError_t e = cudaSuccess;
    if (!smem_configured((const void*)fn, (int)smem)) e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    dim3 grid(vl.ntiles * NDIR, (a.nbands + BPC * nbg - 1) / (BPC * nbg), vl.nk * vl.ns);
    return launch_dependent(fn, grid, NT, smem, st, vl, a, nbg);
}

// The default shape of a table row (variant 0): run_project with its thread count and tiling in the last
// places.
template <int POL, int Q, int CH, int NBG, int PF, int MINB, int NT, int TP>
static cudaError_t run_project_default(const View& v, const ProjArgs& a, cudaStream_t st, View* used) {
    if constexpr (POL == P_PAIR) {
        return run_project<POL, Q, CH, NBG, PF, MINB, 0, 1, NT, TP, true, true>(v, a, st, used);
    } else {
        constexpr int BPC = (NT / 32) * (32 / Q) * LaneBands<POL>::value;
        const int nbg = balanced_groups(NBG, BPC, a.nbands, (int64_t)v.ntiles * v.nk * v.ns, MINB * sm_count());
        if (nbg > NBG / 2) return run_project<POL, Q, CH, NBG, PF, MINB, 0, 1, NT, TP>(v, a, st, used);
        if (nbg > 1) return run_project<POL, Q, CH, NBG / 2, PF, MINB, 0, 1, NT, TP>(v, a, st, used);
        return run_project<POL, Q, CH, 1, PF, MINB, 0, 1, NT, TP>(v, a, st, used);
    }
}

template <int POL, int Q, int CH, int NBG, int PF, int MINB = 2, int NT = CTA>
static cudaError_t run_project_batch(const BatchLaunch& b, cudaStream_t st) {
    size_t smem = TILE * sizeof(int) + (size_t)TILE_PAD * phi_row_bytes(POL, b.maxM);
    cudaError_t e = cudaSuccess;
    auto fn = k_project_batch<POL, Q, CH, NBG, PF, MINB, NT>;
    if (!smem_configured((const void*)fn, (int)smem)) e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    int per_sm = 0, nsm = 0, dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, NT, smem);
    if (e != cudaSuccess) return e;
    e = cudaMemsetAsync(b.counter, 0, sizeof(int), st);
    if (e != cudaSuccess) return e;
    int grid = std::max(1, std::min(per_sm * nsm, b.nitems));
    fn<<<grid, NT, smem, st>>>(b.views, b.args, b.items, b.nitems, b.counter);
    return cudaGetLastError();
}

// The default shape of a table row for the batched launch (always the TILE tiling).
template <int POL, int Q, int CH, int NBG, int PF, int MINB, int NT, int TP>
static cudaError_t run_project_batch_default(const BatchLaunch& b, cudaStream_t st) {
    return run_project_batch<POL, Q, CH, NBG, PF, MINB, NT>(b, st);
}

// Launches of one arithmetic policy's shapes (project_pair.cu, project_f32.cu): variant 0 is the default.
cudaError_t project_pair(const View& v, const ProjArgs& a, int variant, cudaStream_t st, View* used);
cudaError_t project_f32(const View& v, const ProjArgs& a, int variant, cudaStream_t st, View* used);
cudaError_t project_pair_batch(const BatchLaunch& b, int variant, cudaStream_t st);
cudaError_t project_f32_batch(const BatchLaunch& b, int variant, cudaStream_t st);

}  // namespace dftu
