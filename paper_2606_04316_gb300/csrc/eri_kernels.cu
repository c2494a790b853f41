// eri_kernels.cu -- AO two-electron integral tiles on the GPU (stage (i) of
// the paper's Sec. 3.3.1 decomposition), McMurchie-Davidson:
//
//   (xy|K|zw) = sum_{ij in X, kl in Y} sum_{h, h'} E^{ij}_{xy,h} (-1)^{|h'|}
//               E^{kl}_{zw,h'} R^K_{h+h'}(rho, P - Q)
//
//   1/r12 (Eq. Coulomb):    R^n_000 = (-2 rho)^n F_n(T) * 2 pi^{5/2} / (p q sqrt(p+q))
//   r12 (for Eq. gaugeInt): R^n_000 = (-2 rho)^n (F_n - F_{n-1})(T) * pi^{5/2} sqrt(p+q) / (p q)^2,
//                           F_{-1}(T) = -(2 T F_0 + e^{-T})  (Gaussian-smeared distance)
//   gauge kernel:  (xy|r_I r_J/r^3|zw) = delta_IJ (xy|1/r|zw) - (xy|d_I d_J r|zw),
//                  the last term shifting the Hermite index of the r12 tensor by e_I + e_J,
//   R^n_{t+1,u,v} = t R^{n+1}_{t-1,u,v} + X_PQ R^{n+1}_{t,u,v}  (same in u, v).
//
// The signs (-1)^{|h'|} are carried by the tensor: R~_g = (-1)^{|g|} R_g is the
// tensor of Q - P, and (-1)^{|h'|} R_{h+h'} = (-1)^{|h|} R~_{h+h'}.
//
// Work layout: a tile is one bra shell pair and up to 32 ket shell pairs of one kind
// (function pairs and primitive pairs alike), so one orientation (the cheaper one; X
// outer, Y inner) and one cut serve it all.  A CTA takes several kets and outer primitive
// pairs ij at a time through four phases: the headers (Boys values, prefactors; one long dependent
// chain each), the Hermite tensors of all inner primitive pairs by the recursion, the
// ket pass T[h][y] = sum_kl sum_h' R~ E', and the bra pass G += E T.
//
// What bounds it: in the split form no single unit.  The multiply-adds of the two passes
// keep the FP32 pipe busy for a sixth to a quarter of the time, shared-memory loads
// their unit for more than half; what is left is the latency of chains of table,
// tensor and coefficient loads at 12 to 16 warps per SM (128 registers), and instruction
// fetch: tiles of both forms interleaved take 131 ms where apart they take 125 (build_tiles).
// Measured without gain: fewer registers and more warps (80: 183 to 214 ms for the integrals of a 24-centre chain instead
// of 179), tensor entries placed to avoid the ket pass's bank conflicts (172 for 169), four
// function pairs per ket item (178 for 173).  In the FP64 form the FP64 pipe bounds it.
// What keeps the work down:
//  * Boxes.  The expansion of a function pair is a product of one-dimensional
//    ones, so only the Hermite functions of its box (FuncPair) contribute, 27 to
//    37 % of all for the pairs of p functions and derivatives.  Both passes
//    run over the box's list only (the other terms are exact zeros).
//  * Twos of primitive pairs.  R and E hold the inner primitive pairs in twos
//    (hi0, hi1, lo0, lo1), so one 16-byte load feeds one packed FP32
//    instruction (fma.rn.f32x2) per operation: half the issue slots of the
//    scalar form, and the two halves are independent chains.  The bra pass
//    packs two function pairs y instead.
//  * Several kets at a time: a small quartet alone leaves most lanes without work.
// Integrals of a 24-centre chain (Coulomb, Gaunt, gauge) 477 -> 171 ms over these and the
// choices at the phases below, 40-centre chain (Coulomb) 322 -> 128, an 18-atom cluster
// 632 -> 208, a class with d shells 671 -> 65; FP64 form, 7-centre chain 39 -> 11.7.
//
// Split form (DF): recursion and both passes in compensated FP32 pairs (x = hi +
// lo, ~48-bit significands): products by the exact-product FMA, sums by the
// error-free two-sum.  FP32 issues 64 times faster than FP64 on this part.
// Tiles the host admitted to the FP32 error budget run in plain FP32.
#include <math.h>

#include <algorithm>
#include <cstdlib>

#include "qdt_internal.cuh"

namespace qdt {

namespace {

constexpr double kPi52 = 17.493418327624862;        // pi^{5/2}
constexpr double kTwoPi52 = 34.986836655249725;     // 2 pi^{5/2}
constexpr double kHalfSqrtPi = 0.88622692545275801;  // sqrt(pi) / 2
constexpr double kBoysInvDelta = 1.0 / kBoysDelta;

static_assert(kBoysNMax <= 15, "constant tables below hold 16 orders");
static_assert(kBoysTaylor == 7, "constant table below holds 1/k for k < 8");

__constant__ double c_inv_int[8] = {0.0, 1.0, 1.0 / 2, 1.0 / 3, 1.0 / 4, 1.0 / 5, 1.0 / 6, 1.0 / 7};
__constant__ double c_odd[16] = {1, 3, 5, 7, 9, 11, 13, 15, 17, 19, 21, 23, 25, 27, 29, 31};
__constant__ double c_inv_odd[16] = {1.0,      1.0 / 3,  1.0 / 5,  1.0 / 7,  1.0 / 9,  1.0 / 11,
                                     1.0 / 13, 1.0 / 15, 1.0 / 17, 1.0 / 19, 1.0 / 21, 1.0 / 23,
                                     1.0 / 25, 1.0 / 27, 1.0 / 29, 1.0 / 31};


__device__ inline void htrip_d(int h, int &t, int &u, int &v) {
    int s = 0;
    while (nherm(s) <= h) ++s;
    int rem = h - (s ? nherm(s - 1) : 0);
    int uv = 0;
    while ((uv + 1) * (uv + 2) / 2 <= rem) ++uv;
    v = rem - uv * (uv + 1) / 2;
    u = uv - v;
    t = s - uv;
}

// A primitive quartet's header in shared memory: entry j (Q - P, then R^n_000) of one
// half of a two of primitive quartets; `st` scalars between entries.
struct HeadF64 {
    double *p;
    int st;
    __device__ double get(int j) const { return p[j * st]; }
    __device__ void set(int j, double v) const { p[j * st] = v; }
    __device__ void zero(int j) const { p[j * st] = 0.0; }
};
struct HeadPair {                       // (hi0, hi1, lo0, lo1)
    float *p;
    int st;
    __device__ float2 get(int j) const { return make_float2(p[j * st], p[j * st + 2]); }
    __device__ void set(int j, float2 v) const { p[j * st] = v.x; p[j * st + 2] = v.y; }
    __device__ void zero(int j) const { set(j, make_float2(0.f, 0.f)); }
};

// F_0..F_nmax at T into entries j0..j0+nmax; returns exp(-T).  Inside the table: Taylor
// expansion of the top order about the nearest grid point (Horner form), then
// the downward recursion.  Beyond it erf(sqrt T) = 1 to double precision, so
// F_0 = sqrt(pi / T) / 2, then the upward recursion.
__device__ __forceinline__ double boys_eval(const double *tab, double T, int nmax, const HeadF64 &H, int j0) {
    const double e = exp(-T);
    if (T < kBoysTMax) {
        const double ti = rint(T * kBoysInvDelta);
        const int i = (int)ti;
        const double md = fma(ti, kBoysDelta, -T);      // -(T - T_i)
        const double *row = tab + (size_t)i * kBoysCols + nmax;
        double f = __ldg(row + kBoysTaylor - 1);
#pragma unroll
        for (int k = kBoysTaylor - 1; k > 0; --k) f = fma(f, md * c_inv_int[k], __ldg(row + k - 1));
        H.set(j0 + nmax, f);
        const double t2 = T + T;
        for (int n = nmax - 1; n >= 0; --n) {
            f = fma(t2, f, e) * c_inv_odd[n];
            H.set(j0 + n, f);
        }
    } else {
        double f = kHalfSqrtPi * rsqrt(T);
        const double inv2t = 0.5 / T;
        H.set(j0, f);
        for (int n = 0; n < nmax; ++n) {
            f = fma(c_odd[n], f, -e) * inv2t;
            H.set(j0 + n + 1, f);
        }
    }
    return e;
}

// Compensated FP32 pair arithmetic.  The intrinsics keep the compiler from
// fusing the rounded product into the following sum.
__device__ __forceinline__ float2 df_split(double x) {
    const float h = __double2float_rn(x);
    return make_float2(h, __double2float_rn(x - (double)h));
}

// The same split by integer operations on the bits (no FP64 instruction):
// hi = the top 24 significand bits of x, lo = the remaining 29 bits rounded to
// FP32.  Magnitudes outside [2^-70, 2^120) take the FP64 route.
__device__ __forceinline__ float2 df_split_bits(double x) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    const unsigned hi32 = (unsigned)(b >> 32), lo32 = (unsigned)b;
    const int e = (int)((hi32 >> 20) & 0x7FF);
    if (e < 1023 - 70 || e >= 1023 + 120) return df_split(x);
    const unsigned sign = hi32 & 0x80000000u;
    const float h = __uint_as_float(sign | ((unsigned)(e - 1023 + 127) << 23) | ((hi32 & 0xFFFFFu) << 3) |
                                    (lo32 >> 29));
    const float scale = __uint_as_float((unsigned)(e - 1075 + 127) << 23);   // 2^(e - 1075) >= 2^-122
    const float l = __fmul_rn(__uint2float_rn(lo32 & 0x1FFFFFFFu), scale);
    return make_float2(h, __uint_as_float(__float_as_uint(l) | sign));
}

__global__ void split_pairs_kernel(const double2 *E, long long n, float4 *E2, float2 *E1) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) {
        const double2 e = E[i];
        const float2 a = df_split(e.x), b = df_split(e.y);
        E2[i] = make_float4(a.x, b.x, a.y, b.y);
        E1[i] = make_float2(a.x, b.x);
    }
}

// EX of one shell pair per CTA: its entries as FP32 pairs (hi, lo), primitive pair by
// primitive pair.
__global__ void bra_entries_kernel(const PairDev *pairs, const double2 *E, float2 *EX) {
    const PairDev p = pairs[blockIdx.x];
    const double *e = reinterpret_cast<const double *>(E + p.eoff);
    float2 *o = EX + 2 * p.eoff;
    for (int i = threadIdx.x; i < p.nbox * p.npp; i += blockDim.x) {
        const int ij = i / p.nbox, k = i - ij * p.nbox;
        o[i] = df_split(e[2 * (k * p.nk2 + (ij >> 1)) + (ij & 1)]);
    }
}

// Header of a primitive quartet in FP64: Q - P, then R^n_000 of the Coulomb tensor
// (n = 0..L) and, for the gauge kernel, of the r12 tensor (n = 0..L+2).
__host__ __device__ inline int header_len(int L, bool gauge) { return gauge ? 2 * L + 7 : L + 4; }

template <bool GAUGE>
__device__ __forceinline__ void quartet_header(const double *boys, const PrimPairDev *pa, const PrimPairDev *pc,
                                               int L, const HeadF64 &H) {
    const double p = pa->p, q = pc->p, s = p + q;
    const double X = pc->P[0] - pa->P[0], Y = pc->P[1] - pa->P[1], Z = pc->P[2] - pa->P[2];
    const double inv_s = 1.0 / s;
    const double rho = p * q * inv_s;
    const double T = rho * fma(X, X, fma(Y, Y, Z * Z));
    H.set(0, X);
    H.set(1, Y);
    H.set(2, Z);
    const double sq = sqrt(s);
    const double d = pa->inv_p * pc->inv_p * inv_s * sq;      // 1 / (p q sqrt(p + q))
    const double m2r = -2.0 * rho;
    double fC = kTwoPi52 * d;
    if (!GAUGE) {
        boys_eval(boys, T, L, H, 3);
        for (int n = 0; n <= L; ++n) {
            H.set(3 + n, H.get(3 + n) * fC);
            fC *= m2r;
        }
    } else {
        const int jR = 4 + L;
        const double e = boys_eval(boys, T, L + 2, H, jR);
        double fR = kPi52 * s * sq * d * d;
        double prev = -fma(T + T, H.get(jR), e);            // F_{-1}
        for (int n = 0; n <= L + 2; ++n) {
            const double cur = H.get(jR + n);
            if (n <= L) {
                H.set(3 + n, cur * fC);
                fC *= m2r;
            }
            H.set(jR + n, (cur - prev) * fR);
            fR *= m2r;
            prev = cur;
        }
    }
}

// ---------------------------------------------------------------------------
// FP32-pair arithmetic (x = hi + lo, ~2^-47 relative per operation) for the
// header of the compensated-FP32 integrals: error-free product and two-sum,
// renormalised.  The intrinsics keep the compiler from contracting the
// rounded operations.
__device__ __forceinline__ float2 pr_add(float2 a, float2 b) {
    const float s = __fadd_rn(a.x, b.x);
    const float bv = __fsub_rn(s, a.x);
    float e = __fadd_rn(__fsub_rn(a.x, __fsub_rn(s, bv)), __fsub_rn(b.x, bv));
    e = __fadd_rn(e, __fadd_rn(a.y, b.y));
    const float t = __fadd_rn(s, e);
    return make_float2(t, __fsub_rn(e, __fsub_rn(t, s)));
}
__device__ __forceinline__ float2 pr_neg(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float2 pr_mul(float2 a, float2 b) {
    const float p = __fmul_rn(a.x, b.x);
    float e = __fmaf_rn(a.x, b.x, -p);
    e = __fmaf_rn(a.x, b.y, e);
    e = __fmaf_rn(a.y, b.x, e);
    const float t = __fadd_rn(p, e);
    return make_float2(t, __fsub_rn(e, __fsub_rn(t, p)));
}
// times a power of two (exact)
__device__ __forceinline__ float2 pr_pow2(float2 a, float f) { return make_float2(a.x * f, a.y * f); }
// 1/a: the FP32 reciprocal y and one Newton step y + y (1 - a y), the residual in pairs
__device__ __forceinline__ float2 pr_rcp(float2 a) {
    const float y = __frcp_rn(a.x);
    const float2 r = pr_add(make_float2(1.f, 0.f), pr_neg(pr_mul(a, make_float2(y, 0.f))));
    return pr_add(make_float2(y, 0.f), make_float2(__fmul_rn(y, r.x), 0.f));
}
// sqrt(a): the FP32 root y and one Newton step y + (a - y^2) / (2 y)
__device__ __forceinline__ float2 pr_sqrt(float2 a) {
    const float y = __fsqrt_rn(a.x);
    const float2 r = pr_add(a, pr_neg(pr_mul(make_float2(y, 0.f), make_float2(y, 0.f))));
    return pr_add(make_float2(y, 0.f), make_float2(__fdiv_rn(r.x, y + y), 0.f));
}
__host__ __device__ constexpr float2 pair_const(double x) { return float2{(float)x, (float)(x - (double)(float)x)}; }
__constant__ float2 c_inv_int_p[8] = {pair_const(0.0),       pair_const(1.0),       pair_const(1.0 / 2),
                                      pair_const(1.0 / 3),   pair_const(1.0 / 4),   pair_const(1.0 / 5),
                                      pair_const(1.0 / 6),   pair_const(1.0 / 7)};
__constant__ float2 c_inv_odd_p[16] = {
    pair_const(1.0),      pair_const(1.0 / 3),  pair_const(1.0 / 5),  pair_const(1.0 / 7),
    pair_const(1.0 / 9),  pair_const(1.0 / 11), pair_const(1.0 / 13), pair_const(1.0 / 15),
    pair_const(1.0 / 17), pair_const(1.0 / 19), pair_const(1.0 / 21), pair_const(1.0 / 23),
    pair_const(1.0 / 25), pair_const(1.0 / 27), pair_const(1.0 / 29), pair_const(1.0 / 31)};

// F_0..F_nmax at T (a pair) into entries j0..j0+nmax as pairs; returns exp(-T).  Inside
// the table: Taylor expansion of the top order about the nearest grid point
// T_i, exp(-T) = exp(-T_i) exp(T_i - T) (|T_i - T| <= 0.025, eight terms), then
// the downward recursion; beyond it F_0 = sqrt(pi / T) / 2 and the upward
// recursion (exp(-T) < 3e-16 F_0 there, so its FP32 value suffices).
__device__ __forceinline__ float2 boys_eval_pairs(const BoysTables &bt, float2 T, int nmax, const HeadPair &H, int j0) {
    if (T.x < (float)kBoysTMax) {
        const int i = min((int)rintf(T.x * (float)kBoysInvDelta), kBoysGrid - 1);
        const float2 md = pr_add(bt.t_pair[i], pr_neg(T));        // T_i - T
        const float2 *row = bt.pair + (size_t)i * kBoysCols + nmax;
        float2 f = row[kBoysTaylor - 1];
#pragma unroll
        for (int k = kBoysTaylor - 1; k > 0; --k) f = pr_add(pr_mul(f, pr_mul(md, c_inv_int_p[k])), row[k - 1]);
        H.set(j0 + nmax, f);
        float2 em = make_float2(1.f, 0.f);
#pragma unroll
        for (int k = 7; k > 0; --k) em = pr_add(make_float2(1.f, 0.f), pr_mul(em, pr_mul(md, c_inv_int_p[k])));
        const float2 e = pr_mul(bt.exp_pair[i], em);
        const float2 t2 = pr_pow2(T, 2.f);
        for (int n = nmax - 1; n >= 0; --n) {
            f = pr_mul(pr_add(pr_mul(t2, f), e), c_inv_odd_p[n]);
            H.set(j0 + n, f);
        }
        return e;
    }
    const float2 e = make_float2(expf(-T.x), 0.f);
    float2 f = pr_mul(pair_const(kHalfSqrtPi), pr_rcp(pr_sqrt(T)));
    const float2 inv2t = pr_pow2(pr_rcp(T), 0.5f);
    H.set(j0, f);
    for (int n = 0; n < nmax; ++n) {
        f = pr_mul(pr_add(pr_mul(f, make_float2((float)(2 * n + 1), 0.f)), pr_neg(e)), inv2t);
        H.set(j0 + n + 1, f);
    }
    return e;
}

// Header of a primitive quartet whose integrals run in compensated FP32 pairs:
// the same quantities as quartet_header computed in FP32 pairs
// (X_PQ and p + q from FP64 sums, the rest in pairs), so the FP64 pipe does four
// additions per quartet instead of the whole header.  Layout as quartet_header.
template <bool GAUGE>
__device__ __forceinline__ void quartet_header_pairs(const double *boys, const PrimPairDev *pa, const PrimPairDev *pc,
                                                     int L, const HeadPair &H) {
    const BoysTables bt = boys_tables(boys);
    const float2 p = df_split_bits(pa->p), q = df_split_bits(pc->p);
    const float2 s = df_split_bits(pa->p + pc->p);
    const float2 X = df_split_bits(pc->P[0] - pa->P[0]), Y = df_split_bits(pc->P[1] - pa->P[1]),
                 Z = df_split_bits(pc->P[2] - pa->P[2]);
    const float2 inv_s = pr_rcp(s);
    const float2 rho = pr_mul(pr_mul(p, q), inv_s);
    const float2 T = pr_mul(rho, pr_add(pr_add(pr_mul(X, X), pr_mul(Y, Y)), pr_mul(Z, Z)));
    H.set(0, X);
    H.set(1, Y);
    H.set(2, Z);
    const float2 sq = pr_sqrt(s);
    const float2 d = pr_mul(pr_mul(pr_mul(df_split_bits(pa->inv_p), df_split_bits(pc->inv_p)), inv_s), sq);
    const float2 m2r = pr_pow2(rho, -2.f);
    float2 fC = pr_mul(pair_const(kTwoPi52), d);
    if (!GAUGE) {
        boys_eval_pairs(bt, T, L, H, 3);
        for (int n = 0; n <= L; ++n) {
            H.set(3 + n, pr_mul(H.get(3 + n), fC));
            fC = pr_mul(fC, m2r);
        }
    } else {
        const int jR = 4 + L;
        const float2 e = boys_eval_pairs(bt, T, L + 2, H, jR);
        float2 fR = pr_mul(pr_mul(pr_mul(pair_const(kPi52), s), sq), pr_mul(d, d));
        float2 prev = pr_neg(pr_add(pr_mul(pr_pow2(T, 2.f), H.get(jR)), e));     // F_{-1}
        for (int n = 0; n <= L + 2; ++n) {
            const float2 cur = H.get(jR + n);
            if (n <= L) {
                H.set(3 + n, pr_mul(cur, fC));
                fC = pr_mul(fC, m2r);
            }
            H.set(jR + n, pr_mul(pr_add(cur, pr_neg(prev)), fR));
            fR = pr_mul(fR, m2r);
            prev = cur;
        }
    }
}

// Header of a primitive quartet whose integrals run in plain FP32 (only the
// high parts are read): the geometry -- X_PQ, 1/(p+q), rho and T = rho |PQ|^2
// -- in FP64, so that T keeps its absolute accuracy (the Boys values are
// sensitive to it), and the Boys values, exp(-T) and the prefactors in FP32
// from the table's FP32 copy (the FP64 Boys evaluation would hold the FP64
// pipe for most of the header).  Layout as quartet_header, as (value, 0) pairs.
__constant__ float c_inv_int_f[8] = {0.f, 1.f, 1.f / 2, 1.f / 3, 1.f / 4, 1.f / 5, 1.f / 6, 1.f / 7};
__constant__ float c_odd_f[16] = {1, 3, 5, 7, 9, 11, 13, 15, 17, 19, 21, 23, 25, 27, 29, 31};
__constant__ float c_inv_odd_f[16] = {1.f,      1.f / 3,  1.f / 5,  1.f / 7,  1.f / 9,  1.f / 11,
                                      1.f / 13, 1.f / 15, 1.f / 17, 1.f / 19, 1.f / 21, 1.f / 23,
                                      1.f / 25, 1.f / 27, 1.f / 29, 1.f / 31};

// F_0..F_nmax at T into entries j0..j0+nmax (FP32; Taylor offset from the FP64 T).
__device__ __forceinline__ void boys_eval_f32(const float *tab, double T, int nmax, const HeadPair &H, int j0) {
    const float Tf = (float)T;
    const float e = expf(-Tf);
    if (T < kBoysTMax) {
        const double ti = rint(T * kBoysInvDelta);
        const float md = (float)fma(ti, kBoysDelta, -T);       // -(T - T_i), exact to FP32 rounding
        const float *row = tab + (size_t)(int)ti * kBoysCols + nmax;
        float f = __ldg(row + kBoysTaylor - 1);
#pragma unroll
        for (int k = kBoysTaylor - 1; k > 0; --k) f = fmaf(f, md * c_inv_int_f[k], __ldg(row + k - 1));
        H.set(j0 + nmax, make_float2(f, 0.f));
        const float t2 = Tf + Tf;
        for (int n = nmax - 1; n >= 0; --n) {
            f = fmaf(t2, f, e) * c_inv_odd_f[n];
            H.set(j0 + n, make_float2(f, 0.f));
        }
    } else {
        float f = (float)kHalfSqrtPi * rsqrtf(Tf);
        const float inv2t = 0.5f / Tf;
        H.set(j0, make_float2(f, 0.f));
        for (int n = 0; n < nmax; ++n) {
            f = fmaf(c_odd_f[n], f, -e) * inv2t;
            H.set(j0 + n + 1, make_float2(f, 0.f));
        }
    }
}

// Coulomb kernel only (the r12 tensor of the gauge kernel takes differences
// F_n - F_{n-1} that lose digits in FP32, measured 13 times the Coulomb kernel's
// error ratio: its plain-FP32 tiles take the high parts of the FP32-pair header).
__device__ __forceinline__ void quartet_header_f32(const double *boys, const PrimPairDev *pa, const PrimPairDev *pc,
                                                   int L, const HeadPair &H) {
    const double p = pa->p, q = pc->p, s = p + q;
    const double X = pc->P[0] - pa->P[0], Y = pc->P[1] - pa->P[1], Z = pc->P[2] - pa->P[2];
    const double inv_s = 1.0 / s;
    const double rho = p * q * inv_s;
    const double T = rho * fma(X, X, fma(Y, Y, Z * Z));
    H.set(0, make_float2((float)X, 0.f));
    H.set(1, make_float2((float)Y, 0.f));
    H.set(2, make_float2((float)Z, 0.f));
    const float d = (float)pa->inv_p * (float)pc->inv_p * (float)inv_s * sqrtf((float)s);    // 1 / (p q sqrt(p + q))
    const float m2r = (float)(-2.0 * rho);
    float fC = (float)kTwoPi52 * d;
    boys_eval_f32(boys_tables(boys).f32, T, L, H, 3);
    for (int n = 0; n <= L; ++n) {
        H.set(3 + n, make_float2(H.get(3 + n).x * fC, 0.f));
        fC *= m2r;
    }
}

// ---------------------------------------------------------------------------
// Packed FP32: one instruction works on two floats, (lower, upper) in 64 bits.
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
    f32x2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
    f32x2 d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
    f32x2 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
// a - b (one rounding: -1 * b is exact)
__device__ __forceinline__ f32x2 sub2(f32x2 a, f32x2 b) { return fma2(b, 0xBF800000BF800000ull, a); }
__device__ __forceinline__ f32x2 pack2(float x, float y) {
    return (f32x2)__float_as_uint(x) | ((f32x2)__float_as_uint(y) << 32);
}
__device__ __forceinline__ float lower2(f32x2 a) { return __uint_as_float((unsigned)a); }
__device__ __forceinline__ float upper2(f32x2 a) { return __uint_as_float((unsigned)(a >> 32)); }

// a b - p for p = fl(a b), exact, two at once: scalar FMAs, which negate an operand
// for free (a packed one would need the negated operand formed first).
__device__ __forceinline__ f32x2 prod_err2(f32x2 a, f32x2 b, f32x2 p) {
    return pack2(__fmaf_rn(lower2(a), lower2(b), -lower2(p)), __fmaf_rn(upper2(a), upper2(b), -upper2(p)));
}

// (ah, al) += a * b in compensated FP32 pairs, two at once: exact product error of
// the high parts plus the cross terms, then the two-sum of the high parts.
__device__ __forceinline__ void df_madd2(ulonglong2 a, ulonglong2 b, f32x2 &ah, f32x2 &al) {
    const f32x2 p = mul2(a.x, b.x);
    f32x2 pe = prod_err2(a.x, b.x, p);
    pe = fma2(a.x, b.y, pe);
    pe = fma2(a.y, b.x, pe);
    const f32x2 t = add2(ah, p);
    const f32x2 bv = sub2(t, ah);
    const f32x2 err = add2(sub2(ah, sub2(t, bv)), sub2(p, bv));
    ah = t;
    al = add2(al, add2(err, pe));
}

// (h, l) += (a, b), two pairs at once, renormalised; without LOW b is not there and l is left as
// the sum of the errors.
template <bool LOW>
__device__ __forceinline__ void pair_add2(f32x2 &h, f32x2 &l, f32x2 a, f32x2 b) {
    const f32x2 t = add2(h, a);
    const f32x2 bv = sub2(t, h);
    const f32x2 err = add2(sub2(h, sub2(t, bv)), sub2(a, bv));
    if (!LOW) {
        h = t;
        l = add2(l, err);
    } else {
        const f32x2 e = add2(err, add2(l, b));
        h = add2(t, e);
        l = sub2(e, sub2(h, t));
    }
}

// x a + cf c in compensated FP32 pairs, renormalised, two at once (one Hermite
// recursion step).
__device__ __forceinline__ ulonglong2 df_rec2(ulonglong2 x, ulonglong2 a, f32x2 cf, ulonglong2 c) {
    const f32x2 p1 = mul2(x.x, a.x);
    f32x2 e1 = prod_err2(x.x, a.x, p1);
    e1 = fma2(x.x, a.y, e1);
    e1 = fma2(x.y, a.x, e1);
    const f32x2 p2 = mul2(cf, c.x);
    f32x2 e2 = prod_err2(cf, c.x, p2);
    e2 = fma2(cf, c.y, e2);
    const f32x2 t = add2(p1, p2);
    const f32x2 bv = sub2(t, p1);
    const f32x2 err = add2(sub2(p1, sub2(t, bv)), sub2(p2, bv));
    const f32x2 lo = add2(err, add2(e1, e2));
    const f32x2 hi = add2(t, lo);
    return make_ulonglong2(hi, sub2(lo, sub2(hi, t)));
}

// Arithmetic of a tile: FP64, compensated FP32 pairs, plain FP32.  Vec holds one
// two of primitive pairs.
enum { kF64 = 0, kDF = 1, kF32 = 2 };
template <int A> struct Arith;
template <> struct Arith<kF64> { typedef double2 Vec; };
template <> struct Arith<kDF> { typedef ulonglong2 Vec; };
template <> struct Arith<kF32> { typedef f32x2 Vec; };

}  // namespace

// ---------------------------------------------------------------- shared plan
// Sizes from the class maxima.  Tables (built once per CTA) and a pool that
// every quartet divides for itself (partition()).
struct Plan {
    int maxLab;
    int nTab;        // Hermite triples tabulated: nherm of the top order
    int nhm;         // nherm(maxLab)
    int nG;          // T row triples tabulated: nherm(maxLab), gauge nherm(maxLab + 2)
    int nLst;        // box entries of all boxes of order <= maxLab: C(maxLab + 6, 6)
    int threads;
    int pool;        // bytes
};

// A ket shell pair of the current tile.
struct KetRef {
    long long eoff, rowoff, col, col_rev;    // col_rev: its column for the transposed block, < 0: none
    int ppoff, id, mir, pad;                 // mir: transposed block into W2
};
constexpr int kMaxKets = kMaxTileKets;

struct Shape {
    int nE, nO, hs, nT, NC;
};
// How the quartets of a tile (one bra pair, kets of one kind) are cut to fit the
// pool: [headers][even tensors][T | odd tensors][G].  T of a group is written after
// the group's recursion has read the odd tensors and read before the next group
// writes them, so the two share their bytes unless T has to last over several runs
// of inner primitive pairs (nkc < nk2).
struct Cut {
    int xch, ych;        // function pairs of X, Y at a time
    int nkc;             // twos of inner primitive pairs at a time
    int nb;              // kets at a time
    int nij, nijH;       // outer primitive pairs per group, per header pass
};
// Device tables of the shell pairs.
struct PairTables {
    const PrimPairDev *pp;
    const double2 *E;
    const float4 *E2;
    const float2 *E1;
    const float2 *EX;
    const FuncPair *fp;
    const PairChunk *ch;
    const double *boys;
};

// What the phases of a tile need to know about it, written once per tile.  It lives
// in shared memory and the phases are functions of their own, so that a phase's
// loops have the registers to themselves (with everything in one function the
// compensated kernel spilled in its inner loops: 201 ms for the integrals of the
// 24-centre chain, 179 with 168 instead of 128 registers, and this way 179 with 128).
struct TileState {
    PairTables tb;
    const FuncPair *fx;          // X's and Y's tables
    const PairChunk *cy, *cx;
    long long eAB;               // AB's first E entry
    int pAB;                     // and primitive pair
    int swap;                    // X is the ket pair, Y the bra pair AB
    int nkets;
    int L, Ltop;                 // Hermite order of the quartet; top order of its tensors
    int nppx, nfpx, nk2x, nchx, nboxx, nppy, nfpy, nk2y, nchy, nhx;
    int nE_C, nO_C;              // entries of the even and odd tensors before the r12 tensor
    Shape sh;
    Cut c;
    int Re, U, T, G;             // byte offsets in shared memory: even tensors, odd tensors, T, G
    KetRef ket[kMaxKets];        // the tile's kets to compute
    int slot, n_use;             // tile index, kets to compute
    // byte offsets of the tables (built once per CTA) and the pool (headers first)
    int o_src, o_trip, o_box, o_hs, o_rows, o_lst, o_pool;
    int nG, nhm;
};

// Shared memory: TileState, tables, pool.  Every function takes its pointers from
// the array itself, so that the compiler sees shared addresses.
extern __shared__ __align__(16) char sm[];
__device__ __forceinline__ TileState &tile_state() { return *reinterpret_cast<TileState *>(sm); }
template <class T> __device__ __forceinline__ T *at_byte(int off) { return reinterpret_cast<T *>(sm + off); }
// A group within the tile: `nb` kets from ket0, outer primitive pairs ih + i0 ..
// + nij of the header pass's nijH from ih, nk twos of inner primitive pairs from k0,
// function pairs x0 .. + xch, chunks c0 .. c1 of Y (y0 .. + ych, row stride yp).
struct Group {
    int ket0, nb, ih, nijH, i0, nij, k0, nk, x0, xch, c0, c1, y0, ych, yp;
};

__host__ __device__ inline int up16(int n) { return (n + 15) & ~15; }
// Tables: recursion sources of R_h (int2[nTab]); Hermite triple h -> t | u << 8 | v <<
// 16 (int[nTab]); per box its first list entry | count << 16 (int[nhm]); Hermite index
// of the sum of two triples (unsigned short[nhm][nG]); Hermite index that component c's T
// row has for h: h, then h + e_I + e_J (unsigned short[7][nhm]); Hermite indices of the boxes' entries (unsigned char[nLst]).
__host__ __device__ inline int table_bytes(const Plan &p, int (&o)[7]) {
    o[0] = up16((int)sizeof(TileState));
    o[1] = o[0] + up16(p.nTab * 8);
    o[2] = o[1] + up16(p.nTab * 4);
    o[3] = o[2] + up16(p.nhm * 4);
    o[4] = o[3] + up16(p.nG * p.nhm * 2);
    o[5] = o[4] + up16(7 * p.nhm * 2);
    o[6] = o[5] + up16(p.nLst);
    return o[6];
}
size_t plan_tables(const Plan &p) {
    int o[7];
    return (size_t)table_bytes(p, o);
}
size_t plan_smem(const Plan &p) { return plan_tables(p) + (size_t)p.pool; }

// Box entries of all boxes of order < n: C(n + 5, 6).
__host__ __device__ constexpr int box_entries_below(int n) {
    return n * (n + 1) * (n + 2) / 6 * ((n + 3) * (n + 4) / 2) / 2 * (n + 5) / 30;
}
static_assert(box_entries_below(1) == 1 && box_entries_below(2) == 7 && box_entries_below(3) == 28 &&
              box_entries_below(4) == 84 && box_entries_below(5) == 210 && box_entries_below(6) == 462 &&
              box_entries_below(7) == 924, "C(n + 5, 6)");

// Recursion source of R_h: direction, h - e_dir, h - 2 e_dir (packed) and the
// coefficient (component - 1) of the latter as a float.
__device__ void build_tables(const Plan &p) {
    int o[7];
    table_bytes(p, o);
    int2 *src = at_byte<int2>(o[0]);
    int *trip = at_byte<int>(o[1]), *box = at_byte<int>(o[2]);
    unsigned short *hs = at_byte<unsigned short>(o[3]);
    unsigned short *rows = at_byte<unsigned short>(o[4]);
    unsigned char *lst = at_byte<unsigned char>(o[5]);
    if (threadIdx.x == 0) {
        TileState &s = tile_state();
        s.o_src = o[0];
        s.o_trip = o[1];
        s.o_box = o[2];
        s.o_hs = o[3];
        s.o_rows = o[4];
        s.nhm = p.nhm;
        s.o_lst = o[5];
        s.o_pool = o[6];
        s.nG = p.nG;
    }
    for (int h = threadIdx.x; h < p.nTab; h += blockDim.x) {
        int t, u, v;
        htrip_d(h, t, u, v);
        trip[h] = t | (u << 8) | (v << 16);
        int dir, c;
        if (t > 0) { dir = 0; c = t; }
        else if (u > 0) { dir = 1; c = u; }
        else { dir = 2; c = v; }
        int i1 = 0, i2 = 0;
        if (h > 0) {
            const int dt = dir == 0, du = dir == 1, dv = dir == 2;
            i1 = hidx(t - dt, u - du, v - dv);
            if (c >= 2) i2 = hidx(t - 2 * dt, u - 2 * du, v - 2 * dv);
        }
        src[h] = make_int2(dir | (i1 << 2) | (i2 << 12), __float_as_int(c >= 2 ? (float)(c - 1) : 0.f));
        if (h < p.nhm) {
            // this box's list: the boxes before it, of lower order and of its own
            int at = box_entries_below(t + u + v);
            for (int q = nherm(t + u + v - 1); q < h; ++q) {
                int a, bb, c2;
                htrip_d(q, a, bb, c2);
                at += box_count(a, bb, c2);
            }
            box[h] = at | (box_count(t, u, v) << 16);
            for (int x = 0; x <= t; ++x)
                for (int y = 0; y <= u; ++y)
                    for (int z = 0; z <= v; ++z) lst[at++] = (unsigned char)hidx(x, y, z);
            unsigned short *row = rows + h;
            row[0] = (unsigned short)h;
            row[p.nhm] = (unsigned short)hidx(t + 2, u, v);
            row[2 * p.nhm] = (unsigned short)hidx(t + 1, u + 1, v);
            row[3 * p.nhm] = (unsigned short)hidx(t + 1, u, v + 1);
            row[4 * p.nhm] = (unsigned short)hidx(t, u + 2, v);
            row[5 * p.nhm] = (unsigned short)hidx(t, u + 1, v + 1);
            row[6 * p.nhm] = (unsigned short)hidx(t, u, v + 2);
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < p.nG * p.nhm; i += blockDim.x) {
        const int g = trip[i % p.nG], h = trip[i / p.nG];
        hs[i] = (unsigned short)hidx((g & 255) + (h & 255), ((g >> 8) & 255) + ((h >> 8) & 255),
                                       (g >> 16) + (h >> 16));
    }
    __syncthreads();
}

// Sizes of a quartet (X outer, Y inner).  Order-0 and even-order tensors need
// nherm(L) entries each, odd orders nherm(L - 1); the r12 tensor has top order L + 2.
__host__ __device__ inline int odd_len(int Ltop) { return Ltop >= 1 ? nherm(Ltop - 1) : 0; }
__host__ __device__ inline Shape quartet_shape(int Lx, int Ly, bool gauge) {
    const int L = Lx + Ly;
    return {nherm(L) + (gauge ? nherm(L + 2) : 0), odd_len(L) + (gauge ? odd_len(L + 2) : 0), header_len(L, gauge),
            t_rows(Lx, gauge), gauge ? 7 : 1};
}

constexpr int kTensorBytes = 112 * 1024;
// Row stride of T and G: even (a packed load takes two y) but no multiple of 4, so
// that lanes on consecutive T rows store to different banks.
__host__ __device__ inline int y_stride(int ych) {
    const int yp = (ych + 1) & ~1;
    return yp & 3 ? yp : yp + 2;
}
// Entry stride of the tensors, in twos of primitive quartets: odd, so that 16-byte
// loads of consecutive entries (the lanes of the ket pass) fall into different banks.
__host__ __device__ inline int q_stride(int q) { return q | 1; }
// (64 bits: the sizes tried for dozens of kets of contractions of dozens of primitives
// exceed 32.)
__host__ __device__ inline long long cut_bytes(const Shape &s, int nk2, int nb, int xch, int ych, int nkc, int nij,
                                               int nijH) {
    const long long col = (long long)nb * nij, qs = (col * nkc) | 1;
    const int yp = y_stride(ych);
    const long long t = col * s.nT * yp * 8, o = s.nO * qs * 16;
    return (long long)s.hs * nb * nijH * nkc * 16 + s.nE * qs * 16 + (nkc < nk2 ? t + o : (t > o ? t : o)) +
           (long long)nb * s.NC * xch * yp * 8;
}
// The cut decides no rounding except where the inner primitive pairs are cut (nkc,
// contractions of dozens of primitives), and that depends on the quartet alone:
// headers and tensors of one outer primitive pair take at most kTensorBytes, half
// of the largest pool.  Several kets, then several outer primitive pairs are taken at a time until
// the ket pass has work for four rounds of the CTA: a small quartet alone leaves
// most lanes of every phase idle and pays each phase's latency for itself.
__host__ __device__ inline Cut partition(const Shape &s, int nppx, int nfpx, int nppy, int nfpy, int nchy, int nkets,
                                         int pool, int threads) {
    Cut c;
    const int nk2y = (nppy + 1) / 2;
    c.xch = nfpx;
    c.ych = nfpy;
    c.nkc = nk2y > 1 ? nk2y : 1;
    c.nb = 1;
    const int nk2 = c.nkc;
    while (c.nkc > 1 && (s.hs + s.nE + s.nO) * 16 > kTensorBytes / c.nkc) c.nkc = (c.nkc + 1) / 2;
    while (cut_bytes(s, nk2, 1, c.xch, c.ych, c.nkc, 1, 1) > pool) {
        if (c.ych > 4) c.ych = (c.ych + 1) / 2;
        else if (c.xch > 4) c.xch = (c.xch + 1) / 2;
        else if (c.ych > 2) c.ych = 2;
        else if (c.xch > 1) c.xch = (c.xch + 1) / 2;
        else break;
    }
    const int np = nppx > 1 ? nppx : 1, items = s.nT * nchy, want = 4 * threads;
    if (c.nkc == nk2 && c.xch == nfpx && c.ych == nfpy) {
        // kets until the ket pass has its four rounds with three outer primitive pairs each:
        // a ket's columns, 3 x 5 twos of two uncontracted-by-three pairs, then sit together
        // (kets first, one outer pair: 179 ms for the integrals of a 24-centre chain and
        // 139 for 40 centres; two 174 and 135, three 172 and 132, all nine 177 and 140)
        const int nij0 = np < 3 ? np : 3;
        int nb = (want + items * nij0 - 1) / (items * nij0);
        const int nbh = (2 * threads + np * nppy - 1) / (np * (nppy > 1 ? nppy : 1));   // two header rounds
        if (nb < nbh) nb = nbh;
        if (nb > nkets) nb = nkets;
        while (nb > 1 && cut_bytes(s, nk2, nb, c.xch, c.ych, c.nkc, nij0, np) > pool) --nb;
        if (nb > 1) {
            const int groups = (nkets + nb - 1) / nb;
            c.nb = (nkets + groups - 1) / groups;
        }
    }
    int nij = (want + items * c.nb - 1) / (items * c.nb);
    if (nij > np) nij = np;
    while (nij > 1 && cut_bytes(s, nk2, c.nb, c.xch, c.ych, c.nkc, nij, c.nb > 1 ? np : nij) > pool) --nij;
    const int groups = (np + nij - 1) / nij;
    c.nij = (np + groups - 1) / groups;
    c.nijH = c.nb > 1 ? np : c.nij;
    if (c.nb == 1 && c.nkc == nk2) {
        const int rest = pool - (int)cut_bytes(s, nk2, 1, c.xch, c.ych, c.nkc, c.nij, 0);
        int h = rest / (s.hs * c.nkc * 16);
        if (h > np) h = np;
        if (h < np) h = h / c.nij * c.nij;
        if (h > c.nij) c.nijH = h;
    }
    return c;
}

// it / d for it d < 2^32 by a multiply-high with ceil(2^32 / d) (d = 1: the identity).
struct FastDiv {
    unsigned d, magic;
    __device__ explicit FastDiv(int n) : d((unsigned)n), magic(n > 1 ? 0xFFFFFFFFu / (unsigned)n + 1u : 0u) {}
    __device__ int div(int it) const { return magic ? (int)__umulhi((unsigned)it, magic) : it; }
};

template <int A> __device__ __forceinline__ const typename Arith<A>::Vec *e_entries(const PairTables &t);
template <> __device__ __forceinline__ const double2 *e_entries<kF64>(const PairTables &t) { return t.E; }
template <> __device__ __forceinline__ const ulonglong2 *e_entries<kDF>(const PairTables &t) {
    return reinterpret_cast<const ulonglong2 *>(t.E2);
}
template <> __device__ __forceinline__ const f32x2 *e_entries<kF32>(const PairTables &t) {
    return reinterpret_cast<const f32x2 *>(t.E1);
}

// One item of the ket pass: T rows are spread over the lanes, a thread sums one
// row for M function pairs of one box,
//   acc[m] = sum_{j in box} sum_kl R~_kl[h + h_j] E^kl_m[j].
// Each R vector loaded serves the M function pairs; the E vectors are the same
// for all lanes on the same chunk.  NK > 0: that many twos of primitive pairs,
// unrolled (5 = two contractions of three primitives), else nk of them.
template <int A, int M, int NK>
__device__ __forceinline__ void ket_item(const typename Arith<A>::Vec *R, int QS, const unsigned short *hs, int nG,
                                         const unsigned char *lst, int cnt, const typename Arith<A>::Vec *E,
                                         int estride, int nk2, int nk, bool odd, float2 (&out)[M],
                                         double (&outd)[M]) {
    typedef typename Arith<A>::Vec Vec;
    const int n = NK > 0 ? NK : nk;
    int o = (int)hs[lst[0] * nG] * QS;
    if constexpr (A == kF64) {
        double a0[M], a1[M];
#pragma unroll
        for (int m = 0; m < M; ++m) a0[m] = a1[m] = 0.0;
        const int full = odd ? n - 1 : n;               // the last two holds one primitive pair
        for (int j = 0; j < cnt; ++j) {
            const Vec *r = R + o;
            if (j + 1 < cnt) o = (int)hs[lst[j + 1] * nG] * QS;
#pragma unroll 4
            for (int p = 0; p < full; ++p) {
                const Vec rv = r[p];
#pragma unroll
                for (int m = 0; m < M; ++m) {
                    const Vec ev = __ldg(E + m * estride + p);
                    a0[m] = fma(rv.x, ev.x, a0[m]);
                    a1[m] = fma(rv.y, ev.y, a1[m]);
                }
            }
            if (odd) {
                const double rv = r[full].x;
#pragma unroll
                for (int m = 0; m < M; ++m)
                    a0[m] = fma(rv, __ldg(reinterpret_cast<const double *>(E + m * estride + full)), a0[m]);
            }
            E += nk2;
        }
#pragma unroll
        for (int m = 0; m < M; ++m) outd[m] = a0[m] + a1[m];
    } else if constexpr (A == kDF) {
        f32x2 ah[M], al[M];
#pragma unroll
        for (int m = 0; m < M; ++m) ah[m] = al[m] = 0;
        for (int j = 0; j < cnt; ++j) {
            const Vec *r = R + o;
            if (j + 1 < cnt) o = (int)hs[lst[j + 1] * nG] * QS;
#pragma unroll
            for (int p = 0; p < (NK > 0 ? NK : 1); ++p) {
                for (int q = p; q < n; q += (NK > 0 ? n : 1)) {
                    const Vec rv = r[q];
#pragma unroll
                    for (int m = 0; m < M; ++m) df_madd2(rv, __ldg(E + m * estride + q), ah[m], al[m]);
                }
            }
            E += nk2;
        }
#pragma unroll
        for (int m = 0; m < M; ++m)
            out[m] = pr_add(make_float2(lower2(ah[m]), lower2(al[m])), make_float2(upper2(ah[m]), upper2(al[m])));
    } else {
        f32x2 a[M];
#pragma unroll
        for (int m = 0; m < M; ++m) a[m] = 0;
        for (int j = 0; j < cnt; ++j) {
            const Vec *r = R + o;
            if (j + 1 < cnt) o = (int)hs[lst[j + 1] * nG] * QS;
#pragma unroll
            for (int p = 0; p < (NK > 0 ? NK : 1); ++p) {
                for (int q = p; q < n; q += (NK > 0 ? n : 1)) {
                    const Vec rv = r[q];
#pragma unroll
                    for (int m = 0; m < M; ++m) a[m] = fma2(rv, __ldg(E + m * estride + q), a[m]);
                }
            }
            E += nk2;
        }
#pragma unroll
        for (int m = 0; m < M; ++m) out[m] = make_float2(lower2(a[m]) + upper2(a[m]), 0.f);
    }
}

template <int A, int M>
__device__ __forceinline__ void ket_store(const typename Arith<A>::Vec *R, int QS, const unsigned short *hs, int nG,
                                          const unsigned char *lst, int cnt, const typename Arith<A>::Vec *E,
                                          int estride, int nk2, int nk, bool odd, bool neg, bool add, char *T,
                                          int at, int plane) {
    float2 s[M];
    double sd[M];
    if (A != kF64 && nk == 5) ket_item<A, M, 5>(R, QS, hs, nG, lst, cnt, E, estride, nk2, nk, odd, s, sd);
    else ket_item<A, M, 0>(R, QS, hs, nG, lst, cnt, E, estride, nk2, nk, odd, s, sd);
#pragma unroll
    for (int m = 0; m < M; ++m) {
        if constexpr (A == kF64) {
            double *t = reinterpret_cast<double *>(T) + at + m;
            const double v = neg ? -sd[m] : sd[m];
            *t = add ? *t + v : v;
        } else {
            float *t = reinterpret_cast<float *>(T) + at + m;
            float2 v = neg ? pr_neg(s[m]) : s[m];
            if (add) v = pr_add(make_float2(t[0], A == kDF ? t[plane] : 0.f), v);
            t[0] = v.x;
            if (A == kDF) t[plane] = v.y;
        }
    }
}

// Headers of a group's primitive quartets: Q - P, Boys values and prefactors.
template <bool GAUGE, int A>
__device__ __noinline__ void header_pass(const Group g) {
    typedef typename Arith<A == kF64 ? kF64 : kDF>::Vec HVec;      // FP64 or pairs
    const TileState &s = tile_state();
    HVec *H = at_byte<HVec>(s.o_pool);
    const KetRef *kets = s.ket + g.ket0;
    const int QH = g.nb * g.nijH * g.nk, hs = s.sh.hs;
    const FastDiv dk(2 * g.nk), dij(g.nijH);
    for (int q = threadIdx.x; q < 2 * QH; q += blockDim.x) {
        const int o = dk.div(q), r = q - o * 2 * g.nk, kl = 2 * g.k0 + r;
        const int bk = dij.div(o), ij = g.ih + o - bk * g.nijH;
        const int pk = kets[bk].ppoff;
        const PrimPairDev *px = s.tb.pp + (s.swap ? pk : s.pAB) + ij, *py = s.tb.pp + (s.swap ? s.pAB : pk) + kl;
        const int at = o * g.nk + (r >> 1);
        if constexpr (A == kF64) {
            const HeadF64 h{reinterpret_cast<double *>(H + at) + (r & 1), 2 * QH};
            if (kl < s.nppy) {
                quartet_header<GAUGE>(s.tb.boys, px, py, s.L, h);
            } else {
                for (int j = 0; j < hs; ++j) h.zero(j);
            }
        } else {
            const HeadPair h{reinterpret_cast<float *>(H + at) + (r & 1), 4 * QH};
            if (kl < s.nppy) {
                if constexpr (A == kF32 && !GAUGE) quartet_header_f32(s.tb.boys, px, py, s.L, h);
                else quartet_header_pairs<GAUGE>(s.tb.boys, px, py, s.L, h);
            } else {
                for (int j = 0; j < hs; ++j) h.zero(j);
            }
        }
    }
}

// Hermite recursion of a group, one auxiliary order per pass; order 0 ends in the
// even tensors.  In FP64 the double-precision units bound it: items (entry, column) are
// spread over all threads without a remainder (columns kept by a thread: 12.3 instead of
// 11.5 ms for the integrals of a 7-centre chain).
template <bool GAUGE>
__device__ __forceinline__ void recursion_f64(const Group &g) {
    typedef double2 Vec;
    const TileState &s = tile_state();
    const Vec *H = at_byte<Vec>(s.o_pool);
    Vec *Re = at_byte<Vec>(s.Re), *Ro = at_byte<Vec>(s.U);
    const int2 *stab = at_byte<int2>(s.o_src);
    const int L = s.L, Ltop = s.Ltop, nE_C = s.nE_C, nO_C = s.nO_C;
    const int Q2 = g.nb * g.nij * g.nk, QS = q_stride(Q2), QH = g.nb * g.nijH * g.nk;
    const FastDiv dq(Q2), db1(g.nij * g.nk);
    const int hskip = (g.nijH - g.nij) * g.nk, hoff = g.i0 * g.nk;
    for (int m = Ltop; m >= 0; --m) {
        const int cC = m <= L ? nherm(L - m) : 0;
        const int cR = GAUGE ? nherm(Ltop - m) : 0;
        Vec *dst = (m & 1) ? Ro : Re;
        const Vec *src = (m & 1) ? Re : Ro;
        const int dR = (m & 1) ? nO_C : nE_C, sR = ((m & 1) ? nE_C : nO_C) * QS;
        const int jC = (3 + m) * QH, jR = (4 + L + m) * QH;
        for (int it = threadIdx.x; it < (cC + cR) * Q2; it += blockDim.x) {
            const int e = dq.div(it);
            const int q = it - e * Q2;
            const int hq = q + hoff + (g.nb > 1 ? db1.div(q) * hskip : 0);
            const bool r12 = GAUGE && e >= cC;
            const int h = r12 ? e - cC : e;
            Vec r;
            if (h == 0) {
                r = H[(r12 ? jR : jC) + hq];
            } else {
                const int2 sw = stab[h];
                const Vec *sp = src + (r12 ? sR : 0) + q;
                const Vec xv = H[(sw.x & 3) * QH + hq];
                const Vec a = sp[((sw.x >> 2) & 1023) * QS];
                const Vec cc = sp[(sw.x >> 12) * QS];
                const double cf = (double)__int_as_float(sw.y);
                r = make_double2(fma(cf, cc.x, xv.x * a.x), fma(cf, cc.y, xv.y * a.y));
            }
            dst[((r12 ? dR : 0) + h) * QS + q] = r;
        }
        __syncthreads();
    }
}

template <int A>
__device__ __forceinline__ typename Arith<A>::Vec rec_step(Arith<kDF>::Vec x, typename Arith<A>::Vec a, float cf,
                                                           typename Arith<A>::Vec c) {
    if constexpr (A == kDF) return df_rec2(x, a, pack2(cf, cf), c);
    else return fma2(x.x, a, mul2(pack2(cf, cf), c));
}

// In FP32 (pairs) the shared-memory loads and the integer work around a step bound it: a
// thread keeps one column (ket, outer primitive pair, two of inner ones) with the Q - P
// that most entries step along, and takes two entries at a time, whose loads and about ten
// dependent operations hide each other.  In the gauge kernel an entry of the Coulomb
// tensor goes with the same entry of the r12 tensor: same sources, same Q - P.  Sources
// whose coefficient is zero are not read.  Integrals of a 24-centre chain 172.6 ms, of an
// 18-atom cluster 205; with items (entry, column) 178.6 and 214.5.
template <bool GAUGE, int A>
__device__ __forceinline__ void recursion_columns(const Group &g) {
    typedef typename Arith<A>::Vec Vec;
    typedef Arith<kDF>::Vec HVec;
    const TileState &s = tile_state();
    const int2 *stab = at_byte<int2>(s.o_src);
    const int L = s.L, Ltop = s.Ltop;
    const int Q2 = g.nb * g.nij * g.nk, QS = q_stride(Q2), QH = g.nb * g.nijH * g.nk;
    // columns of the group in runs of at most the CTA's threads, W threads to a column
    const int qn = min(Q2, (int)blockDim.x), W = (int)blockDim.x / qn;
    const int e0 = (int)threadIdx.x / qn, qt = (int)threadIdx.x - e0 * qn;
    const FastDiv db1(g.nij * g.nk);
    const int dE = GAUGE ? s.nE_C * QS : 0, dO = GAUGE ? s.nO_C * QS : 0;       // the r12 tensor's parts
    auto head = [](HVec v) -> Vec {
        if constexpr (A == kF32) return v.x;
        else return v;
    };
    for (int q0 = 0; q0 < Q2; q0 += qn) {
        const int q = q0 + qt;
        const bool mine = q < Q2 && e0 < W;
        const HVec *Hq = at_byte<HVec>(s.o_pool) +
                         (mine ? q + g.i0 * g.nk + (g.nb > 1 ? db1.div(q) * (g.nijH - g.nij) * g.nk : 0) : 0);
        const HVec X0 = *Hq;                    // most entries step along x
        for (int m = Ltop; m >= 0; --m) {
            const int cC = m <= L ? nherm(L - m) : 0;                   // Coulomb tensor (with GAUGE: the second one)
            const int cR = GAUGE ? nherm(Ltop - m) : cC;
            Vec *dp = at_byte<Vec>((m & 1) ? s.U : s.Re) + q;
            const Vec *sp = at_byte<Vec>((m & 1) ? s.Re : s.U) + q;
            const int dR = (m & 1) ? dO : dE, sR = (m & 1) ? dE : dO;
            if (m == Ltop) {            // one entry; there is no order above to read
                if (mine && e0 == 0) dp[dR] = head(Hq[(GAUGE ? 4 + L + m : 3 + m) * QH]);
            } else if (mine) {
#pragma unroll 1
                for (int h = e0; h < cR; h += 2 * W) {
                    const int h2 = h + W;
                    const bool two = h2 < cR;
                    const int2 w1 = stab[h], w2 = stab[two ? h2 : h];
                    const int a1 = ((w1.x >> 2) & 1023) * QS, b1 = (w1.x >> 12) * QS;
                    const int a2 = ((w2.x >> 2) & 1023) * QS, b2 = (w2.x >> 12) * QS;
                    HVec x1 = X0, x2 = X0;
                    if (w1.x & 3) x1 = Hq[(w1.x & 3) * QH];
                    if (w2.x & 3) x2 = Hq[(w2.x & 3) * QH];
                    const float f1 = __int_as_float(w1.y), f2 = __int_as_float(w2.y);
                    Vec r1 = sp[sR + a1], r2 = sp[sR + a2], c1 = r1, c2 = r2;     // coefficient 0: any value
                    if (w1.y) c1 = sp[sR + b1];
                    if (w2.y) c2 = sp[sR + b2];
                    r1 = rec_step<A>(x1, r1, f1, c1);
                    r2 = rec_step<A>(x2, r2, f2, c2);
                    if (h == 0) r1 = head(Hq[(GAUGE ? 4 + L + m : 3 + m) * QH]);
                    dp[dR + h * QS] = r1;
                    if (two) dp[dR + h2 * QS] = r2;
                    if (GAUGE && h < cC) {
                        r1 = sp[a1], r2 = sp[a2], c1 = r1, c2 = r2;
                        if (w1.y) c1 = sp[b1];
                        if (w2.y) c2 = sp[b2];
                        r1 = rec_step<A>(x1, r1, f1, c1);
                        r2 = rec_step<A>(x2, r2, f2, c2);
                        if (h == 0) r1 = head(Hq[(3 + m) * QH]);
                        dp[h * QS] = r1;
                        if (h2 < cC) dp[h2 * QS] = r2;
                    }
                }
            }
            __syncthreads();
        }
    }
}

template <bool GAUGE, int A>
__device__ __noinline__ void recursion_pass(const Group g) {
    if constexpr (A == kF64) recursion_f64<GAUGE>(g);
    else recursion_columns<GAUGE, A>(g);
}

// Ket pass of a group: T rows h < nhx from the Coulomb tensor, then (gauge) rows
// g = 4.. from the r12 tensor.
template <bool GAUGE, int A>
__device__ __noinline__ void ket_pass(const Group g) {
    typedef typename Arith<A>::Vec Vec;
    const TileState &s = tile_state();
    const int nT = s.sh.nT, nhx = s.nhx, nk2y = s.nk2y;
    const int nrows = g.nb * g.nij * nT, tplane = nrows * g.yp;
    const int QS = q_stride(g.nb * g.nij * g.nk);
    const bool odd = (s.nppy & 1) && g.k0 + g.nk == nk2y;
    const Vec *Re = at_byte<Vec>(s.Re);
    const Vec *E0 = e_entries<A>(s.tb);
    char *T = at_byte<char>(s.T);
    const int *trip = at_byte<int>(s.o_trip), *box = at_byte<int>(s.o_box);
    const unsigned short *hs = at_byte<unsigned short>(s.o_hs);
    const unsigned char *lst = at_byte<unsigned char>(s.o_lst);
    const int nG = s.nG;
    const bool swap = s.swap != 0;
    const FastDiv drow(nrows), dT(nT), dnij(g.nij);
    for (int it = threadIdx.x; it < nrows * (g.c1 - g.c0); it += blockDim.x) {
        const int ci = drow.div(it), row = it - ci * nrows;
        const int o = dT.div(row), hh = row - o * nT;
        const int4 kc = __ldg(reinterpret_cast<const int4 *>(s.cy + g.c0 + ci));
        const PairChunk k{kc.x, kc.y, kc.z, kc.w};
        const bool r12 = GAUGE && hh >= nhx;
        const int gh = r12 ? hh - nhx + 4 : hh;
        const int tr = trip[gh];
        const bool neg = ((tr ^ (tr >> 8) ^ (tr >> 16)) & 1) != 0;      // |gh| odd
        const int bx = box[k.box], cnt = bx >> 16;
        const Vec *R = Re + (r12 ? s.nE_C : 0) * QS + o * g.nk;
        const long long ey = swap ? s.eAB : s.ket[g.ket0 + dnij.div(o)].eoff;
        const Vec *E = E0 + ey + (k.off * nk2y + g.k0);
        const int at = row * g.yp + k.k0 - g.y0;
        if (k.m == 2)
            ket_store<A, 2>(R, QS, hs + gh, nG, lst + (bx & 0xffff), cnt, E, cnt * nk2y, nk2y, g.nk, odd, neg,
                            g.k0 > 0, T, at, tplane);
        else
            ket_store<A, 1>(R, QS, hs + gh, nG, lst + (bx & 0xffff), cnt, E, 0, nk2y, g.nk, odd, neg, g.k0 > 0, T,
                            at, tplane);
    }
}

// Bra pass of a group, outer primitive pairs in order (neither the group nor the tile
// changes a rounding):
//   G[c][x][y] += sum_ij sum_{j in box x} E^{ij}_x[j] T[ij][row(c, h_j)][y].
// In the FP32 forms a thread sums the box of one outer primitive pair in the tile's arithmetic
// and adds it to G, which is a pair in both, with the rounding errors kept (pair_add2): one sum
// over all outer pairs lost digits with the length of the contraction (16 primitives per shell:
// plain FP32 within 1.1e-6 Q_A Q_C instead of 8.9e-8, pairs 3.7e-13 instead of 2.6e-14) for 1 to
// 3 % less time (integrals of a 24-centre chain 168.9 ms instead of 171.2, 40 centres 125.2
// instead of 127.9).
// A thread sums one component of TX function pairs x of one box and TY twos of function
// pairs y (FP64: TY function pairs).  With TX = TY = 2 every E and T value loaded serves
// two sums; with 1 there are four times as many items, for quartets so small that the
// larger tile leaves most of the CTA without work (bra_pass chooses).
template <bool GAUGE, int A, int TX, int TY>
__device__ __forceinline__ void bra_tiles(const Group &g) {
    typedef typename Arith<A>::Vec Vec;
    constexpr int NC = GAUGE ? 7 : 1, W = A == kF64 ? 1 : 2;            // function pairs y per step
    const TileState &s = tile_state();
    const int nT = s.sh.nT, nk2x = s.nk2x, nij = g.nij, yp = g.yp, nb = g.nb, xch = g.xch;
    const int tplane = nb * nij * nT * yp, r12off = s.nhx - 4;
    const int gc = xch * yp, gplane = nb * NC * gc;
    const int ny = (g.ych + W * TY - 1) / (W * TY), nx = TX > 1 ? s.nchx : xch;
    const Vec *E0 = e_entries<A>(s.tb);
    const float2 *EX = s.tb.EX;
    const int nboxx = s.nboxx;
    const int4 *cx = reinterpret_cast<const int4 *>(s.cx);
    const int2 *fx = reinterpret_cast<const int2 *>(s.fx) + g.x0;
    const bool swap = s.swap != 0;
    const long long eAB = s.eAB;
    const int *box = at_byte<int>(s.o_box);
    const unsigned char *lst0 = at_byte<unsigned char>(s.o_lst);
    const unsigned short *rows = at_byte<unsigned short>(s.o_rows);
    const int nhm = s.nhm, ij0 = g.ih + g.i0;
    char *const Gp = at_byte<char>(s.G), *const Tp = at_byte<char>(s.T);
    const FastDiv dy(ny), dx(nx), db(nb);
#pragma unroll 1
    for (int it = threadIdx.x; it < NC * nb * nx * ny; it += blockDim.x) {
        const int r0 = dy.div(it), r1 = dx.div(r0), c = NC > 1 ? db.div(r1) : 0;
        const int y = (it - r0 * ny) * W * TY, xi = r0 - r1 * nx, bk = r1 - c * nb;
        int x, m, bx, off;
        if (TX > 1) {
            const int4 k = __ldg(cx + xi);
            x = k.x;
            m = k.y;
            bx = k.z;
            off = k.w;
        } else {
            const int2 f = __ldg(fx + xi);
            x = xi;
            m = 1;
            bx = f.x >> 16;
            off = f.y;
        }
        const int bb = box[bx], cnt = bb >> 16;
        const unsigned char *lst = lst0 + (bb & 0xffff);
        const unsigned short *row = rows + c * nhm;
        const int rowoff = c ? r12off : 0;
        const long long eoff = swap ? s.ket[g.ket0 + bk].eoff : eAB;
        const int x1 = TX > 1 && m > 1 ? cnt : 0;                      // the second x's entries
        const int y1 = TY > 1 ? min(W, yp - W - y) : 0;                // the second y, or one in the row
        const int gi = (bk * NC + c) * gc + x * yp + y;
        if constexpr (A == kF64) {
            double sum[TX][TY];
            double *go = reinterpret_cast<double *>(Gp) + gi;
#pragma unroll
            for (int p = 0; p < TX; ++p)
#pragma unroll
                for (int q = 0; q < TY; ++q) sum[p][q] = go[(p < m ? p : 0) * yp + (q ? y1 : 0)];
#pragma unroll 1
            for (int i = 0; i < nij; ++i) {
                const double *e =
                    reinterpret_cast<const double *>(E0 + eoff + off * nk2x + ((ij0 + i) >> 1)) + ((ij0 + i) & 1);
                const double *t = reinterpret_cast<const double *>(Tp) + ((bk * nij + i) * nT + rowoff) * yp + y;
#pragma unroll 2
                for (int j = 0; j < cnt; ++j) {
                    const double *tr = t + row[lst[j]] * yp;
                    double tv[TY];
#pragma unroll
                    for (int q = 0; q < TY; ++q) tv[q] = tr[q ? y1 : 0];
#pragma unroll
                    for (int p = 0; p < TX; ++p) {
                        const double ev = __ldg(e + 2 * (p ? x1 : 0) * nk2x);
#pragma unroll
                        for (int q = 0; q < TY; ++q) sum[p][q] = fma(ev, tv[q], sum[p][q]);
                    }
                    e += 2 * nk2x;
                }
            }
#pragma unroll
            for (int p = 0; p < TX; ++p)
#pragma unroll
                for (int q = 0; q < TY; ++q)
                    if (p < m && (q == 0 || y + 1 < g.ych)) go[p * yp + q] = sum[p][q];
        } else {
            float *go = reinterpret_cast<float *>(Gp) + gi;
#pragma unroll 1
            for (int i = 0; i < nij; ++i) {
                const float2 *e = EX + 2 * eoff + (ij0 + i) * nboxx + off;
                const float *t = reinterpret_cast<const float *>(Tp) + ((bk * nij + i) * nT + rowoff) * yp + y;
                f32x2 ah[TX][TY], al[TX][TY];
#pragma unroll
                for (int p = 0; p < TX; ++p)
#pragma unroll
                    for (int q = 0; q < TY; ++q) ah[p][q] = al[p][q] = 0;
#pragma unroll 2
                for (int j = 0; j < cnt; ++j) {
                    const float *tr = t + row[lst[j]] * yp;
                    f32x2 th[TY], tl[TY];
#pragma unroll
                    for (int q = 0; q < TY; ++q) {
                        th[q] = *reinterpret_cast<const f32x2 *>(tr + (q ? y1 : 0));
                        if (A == kDF) tl[q] = *reinterpret_cast<const f32x2 *>(tr + tplane + (q ? y1 : 0));
                    }
#pragma unroll
                    for (int p = 0; p < TX; ++p) {
                        const float2 ep = __ldg(e + (p ? x1 : 0));
                        const ulonglong2 ev = make_ulonglong2(pack2(ep.x, ep.x), pack2(ep.y, ep.y));
#pragma unroll
                        for (int q = 0; q < TY; ++q) {
                            if constexpr (A == kDF) df_madd2(ev, make_ulonglong2(th[q], tl[q]), ah[p][q], al[p][q]);
                            else ah[p][q] = fma2(ev.x, th[q], ah[p][q]);
                        }
                    }
                    ++e;
                }
#pragma unroll
                for (int p = 0; p < TX; ++p)
#pragma unroll
                    for (int q = 0; q < TY; ++q)
                        if (p < m && (q == 0 || y + 2 < g.ych)) {
                            f32x2 *gh = reinterpret_cast<f32x2 *>(go + p * yp + 2 * q);
                            f32x2 *gl = reinterpret_cast<f32x2 *>(go + gplane + p * yp + 2 * q);
                            pair_add2<A == kDF>(*gh, *gl, ah[p][q], al[p][q]);
                        }
            }
        }
    }
}

template <bool GAUGE, int A>
__device__ __noinline__ void bra_pass(const Group g) {
    constexpr int NC = GAUGE ? 7 : 1, W = A == kF64 ? 1 : 2;
    const TileState &s = tile_state();
    // rounds of the CTA times instructions per term, about 72 against 26 in FP32 pairs (never
    // the larger tile: integrals of a 40-centre chain 131 -> 134 ms, of a class with d shells
    // 63 -> 66, of a 24-centre chain with the gauge term the same)
    const int n1 = NC * g.nb * g.xch * ((g.ych + W - 1) / W), n2 = NC * g.nb * s.nchx * ((g.ych + 2 * W - 1) / (2 * W));
    const int nt = blockDim.x, r1 = (n1 + nt - 1) / nt, r2 = (n2 + nt - 1) / nt;
    if (g.xch == s.nfpx && 11 * r2 < 4 * r1) bra_tiles<GAUGE, A, 2, 2>(g);
    else bra_tiles<GAUGE, A, 1, 1>(g);
}

// Describes the tile of bra pair AB and `nkets` ket pairs TileState::ket of CD's kind (X = CD
// when swap) to the phases; ends with a barrier.
__device__ __noinline__ void set_tile(const PairTables &tb, const PairDev &AB, const PairDev &CD, bool swap, bool gauge,
                                      int nkets, int pool) {
    const PairDev &X = swap ? CD : AB, &Y = swap ? AB : CD;
    if (threadIdx.x == 0) {
        TileState &s = tile_state();
        s.tb = tb;
        s.fx = tb.fp + X.fpoff;
        s.cy = tb.ch + Y.choff;
        s.cx = tb.ch + X.choff;
        s.nchx = X.nch;
        s.nboxx = X.nbox;
        s.eAB = AB.eoff;
        s.pAB = AB.ppoff;
        s.swap = swap;
        s.nkets = nkets;
        s.L = X.Lab + Y.Lab;
        s.Ltop = s.L + (gauge ? 2 : 0);
        s.nppx = X.npp;
        s.nfpx = X.nfp;
        s.nk2x = X.nk2;
        s.nppy = Y.npp;
        s.nfpy = Y.nfp;
        s.nk2y = Y.nk2;
        s.nchy = Y.nch;
        s.nhx = nherm(X.Lab);
        s.nE_C = nherm(s.L);
        s.nO_C = odd_len(s.L);
        const Shape sh = quartet_shape(X.Lab, Y.Lab, gauge);
        const Cut c = partition(sh, X.npp, X.nfp, Y.npp, Y.nfp, Y.nch, nkets, pool, (int)blockDim.x);
        s.sh = sh;
        s.c = c;
        const int qs = q_stride(c.nb * c.nij * c.nkc), tbytes = c.nb * c.nij * sh.nT * y_stride(c.ych) * 8;
        const int obytes = sh.nO * qs * 16;
        const bool runs = c.nkc < Y.nk2;
        s.Re = s.o_pool + sh.hs * c.nb * c.nijH * c.nkc * 16;
        s.U = s.Re + sh.nE * qs * 16;
        s.T = runs ? s.U + obytes : s.U;
        s.G = s.U + (runs ? tbytes + obytes : max(tbytes, obytes));
    }
    __syncthreads();
}

// The blocks (X|Y) of the tile, some kets and chunks at a time; emit(g, value) is
// called by all threads once a group's results stand in shared memory, value(ket, c,
// x, y) being component c of function pairs x, y (sorted order, relative to the
// chunk).
// Components: 0 Coulomb; gauge kernel 1..6: (xy|d_I d_J r|zw), IJ = xx, xy, xz, yy, yz, zz.
template <bool GAUGE, int A, class Emit>
__device__ __forceinline__ void quartet_blocks(Emit emit) {
    constexpr int NC = GAUGE ? 7 : 1;
    const TileState &s = tile_state();
    Group g;
    for (g.ket0 = 0; g.ket0 < s.nkets; g.ket0 += s.c.nb) {
        g.nb = min(s.c.nb, s.nkets - g.ket0);
        for (g.c0 = 0; g.c0 < s.nchy; g.c0 = g.c1) {
            g.y0 = s.cy[g.c0].k0;
            g.c1 = s.nchy;
            g.ych = s.nfpy - g.y0;
            if (g.ych > s.c.ych) {
                g.c1 = g.c0;
                while (s.cy[g.c1].k0 + s.cy[g.c1].m - g.y0 <= s.c.ych) ++g.c1;
                g.ych = s.cy[g.c1 - 1].k0 + s.cy[g.c1 - 1].m - g.y0;
            }
            g.yp = y_stride(g.ych);
            for (g.x0 = 0; g.x0 < s.nfpx; g.x0 += s.c.xch) {
                g.xch = min(s.c.xch, s.nfpx - g.x0);
                const int gplane = g.nb * NC * g.xch * g.yp;    // FP32 pairs: high parts, then low parts
                double *G = at_byte<double>(s.G);
                for (int i = threadIdx.x; i < gplane; i += blockDim.x) G[i] = 0.0;
                for (g.ih = 0; g.ih < s.nppx; g.ih += s.c.nijH) {
                    g.nijH = min(s.c.nijH, s.nppx - g.ih);
                    for (g.k0 = 0; g.k0 < s.nk2y; g.k0 += s.c.nkc) {
                        g.nk = min(s.c.nkc, s.nk2y - g.k0);
                        __syncthreads();                    // the last recursion has read the headers
                        header_pass<GAUGE, A>(g);
                        __syncthreads();
                        for (g.i0 = 0; g.i0 < g.nijH; g.i0 += s.c.nij) {
                            g.nij = min(s.c.nij, g.nijH - g.i0);
                            if (s.Ltop & 1) __syncthreads();    // T, which the odd tensors overwrite, has been read
                            recursion_pass<GAUGE, A>(g);     // ends with a barrier
                            ket_pass<GAUGE, A>(g);
                            __syncthreads();
                            // T is complete with the last run of inner primitive pairs (with several, nijH == nij)
                            if (g.k0 + g.nk == s.nk2y) bra_pass<GAUGE, A>(g);
                        }
                    }
                }
                __syncthreads();
                emit(g, [&](int bk, int cc, int x, int y) -> double {
                    const int i = ((bk * NC + cc) * g.xch + x) * g.yp + y;
                    if constexpr (A == kF64) return G[i];
                    const float *f = reinterpret_cast<const float *>(G);
                    return (double)f[i] + (double)f[gplane + i];
                });
                __syncthreads();
            }
        }
    }
}

// Screened rows as a persistent kernel: every CTA builds its tables once, then
// takes tiles (bra shell pair x kets of one kind, from the bucket list) from the
// shared counter until none are left.  A tile's parameter set comes from prms[req],
// so one launch can mix the tiles of several transformations.
template <bool GAUGE, bool DF>
__global__ void __launch_bounds__(256, 2) eri_rows_kernel(const EriParams *prms, const EriTask *tasks,
                                                          int *queue, Plan pl) {
    build_tables(pl);
    TileState &s = tile_state();
    const int nt = queue[1];
    const int ij_of[3][3] = {{0, 1, 2}, {1, 3, 4}, {2, 4, 5}};
    for (;;) {
        if (threadIdx.x == 0) s.slot = atomicAdd(queue, 1);
        __syncthreads();
        const int t = s.slot;
        if (t >= nt) break;
        const EriTask tk = tasks[t];
        const EriParams &prm = prms[tk.req];
        // the tile's kets that are computed here, in list order (first warp)
        if (threadIdx.x < 32) {
            bool use = (int)threadIdx.x < tk.k1 - tk.k0;
            KetRef k{};
            if (use) {
                const int kp = prm.bucket[tk.k0 + threadIdx.x];
                const int cd = prm.ket_sp[kp];
                const PairDev &p = prm.pairs[cd];
                k.id = cd;
                k.eoff = p.eoff;
                k.rowoff = p.rowoff;
                k.ppoff = p.ppoff;
                k.col = prm.ket_col[kp];
                // (CD|AB) also kept?  Then one block serves both (EriParams::sym):
                // rev writes it at (cd, ab) of W, mir into W2 for a later batch
                const bool both = prm.sym && cd != tk.bra_sp && prm.ket_pos[tk.bra_sp] < prm.prefix[cd];
                bool rev = both;
                if (both && prm.sym == 2) {
                    const int bp = prm.bra_pos[cd];
                    if (bp < prm.b0) use = false;        // its transpose came from W2 of CD's batch
                    rev = bp < prm.b1;
                    k.mir = !rev;
                }
                if (rev && cd < tk.bra_sp) use = false;
                k.col_rev = rev ? prm.ket_col[prm.ket_pos[tk.bra_sp]] : -1;
            }
            const unsigned mask = __ballot_sync(0xffffffffu, use);
            if (use) s.ket[__popc(mask & ((1u << threadIdx.x) - 1u))] = k;
            if (threadIdx.x == 0) s.n_use = __popc(mask);
        }
        __syncthreads();
        const int nkets = s.n_use;
        if (nkets > 0) {
            const PairDev &AB = prm.pairs[tk.bra_sp];
            const PairDev &CD = prm.pairs[s.ket[0].id];     // all kets of the tile are of its kind
            // contract the orientation with fewer multiply-adds; swapped -> the block is (CD|AB)
            const bool swap = orient_madds(CD, AB, GAUGE) < orient_madds(AB, CD, GAUGE);
            set_tile(PairTables{prm.pp, prm.E, prm.E2, prm.E1, prm.EX, prm.fp, prm.ch, prm.boys}, AB, CD, swap, GAUGE, nkets,
                     pl.pool);
            auto emit = [&](const Group &g, auto value) {
                const FuncPair *fpx = s.fx + g.x0;
                const FuncPair *fpy = prm.fp + (swap ? AB.fpoff : CD.fpoff) + g.y0;
                const long long ldw = prm.ldw, ldwc = prm.ldwc, row0 = prm.row0, rowAB = AB.rowoff - row0;
                const bool wc = prm.with_coulomb != 0;
                const FastDiv dy(g.ych), dx(g.xch);
                for (int idx = threadIdx.x; idx < g.nb * g.xch * g.ych; idx += blockDim.x) {
                    const int bx = dy.div(idx), yy = idx - bx * g.ych, bk = dx.div(bx), xx = bx - bk * g.xch;
                    const int fx = fpx[xx].fp & 0xffff, fy = fpy[yy].fp & 0xffff;
                    const int a = swap ? fy : fx;                // bra function pair
                    const int c = swap ? fx : fy;                // ket function pair
                    const KetRef &k = s.ket[g.ket0 + bk];
                    const double C = value(bk, 0, xx, yy);
                    double hc[6];
                    if (GAUGE)
#pragma unroll
                        for (int j = 0; j < 6; ++j) hc[j] = value(bk, j + 1, xx, yy);
                    // the block's entry into row `r`, column `k` of an output
                    // (gauge: rows (r, I), columns (k, J); K_IJ is symmetric, so the
                    // transposed entry needs no index change)
                    auto put = [&](double *Wo, long long ldo, double *Wco, long long ldco, long long r, long long kc) {
                        if (!GAUGE) {
                            Wo[r * ldo + kc] = C;
                        } else {
#pragma unroll
                            for (int I = 0; I < 3; ++I)
#pragma unroll
                                for (int J = 0; J < 3; ++J)
                                    Wo[(r * 3 + I) * ldo + kc * 3 + J] = (I == J ? C : 0.0) - hc[ij_of[I][J]];
                            if (wc) Wco[r * ldco + kc] = C;
                        }
                    };
                    put(prm.W, ldw, prm.Wc, ldwc, rowAB + a, k.col + c);
                    // the same integrals at (cd, ab): rows of CD, columns of AB
                    if (k.col_rev >= 0) put(prm.W, ldw, prm.Wc, ldwc, k.rowoff + c - row0, k.col_rev + a);
                    if (k.mir) put(prm.W2, prm.ldw2, prm.Wc2, prm.ldwc2, k.rowoff + c - prm.row2,
                                   prm.col2[tk.bra_sp] + a);
                }
            };
            if constexpr (DF) {
                if (tk.f32) quartet_blocks<GAUGE, kF32>(emit);
                else quartet_blocks<GAUGE, kDF>(emit);
            } else {
                quartet_blocks<GAUGE, kF64>(emit);
            }
        }
        __syncthreads();
    }
}

// Plan for a class: the smallest shared-memory tier (so the most CTAs per SM)
// that holds the class's largest quartet uncut, one outer primitive pair at a
// time with the headers of all; at most what its small quartets can use.
Plan eri_plan(int maxnfp, int maxLab, int maxnpp, bool gauge) {
    struct Tier { int kb, threads; };
    const Tier tiers[4] = {{56, 128}, {75, 128}, {112, 256}, {224, 256}};
    Plan p{};
    p.maxLab = maxLab;
    p.nTab = nherm(2 * maxLab + (gauge ? 2 : 0));
    p.nhm = nherm(maxLab);
    p.nG = nherm(maxLab + (gauge ? 2 : 0));
    p.nLst = box_entries_below(maxLab + 1);
    const int npp = std::max(maxnpp, 1), nfp = std::max(maxnfp, 1);
    const Shape s = quartet_shape(maxLab, maxLab, gauge);
    const int nk2 = std::max(1, std::min((npp + 1) / 2, kTensorBytes / ((s.hs + s.nE + s.nO) * 16)));
    const long long tables = (long long)plan_tables(p);
    auto bytes = [&](long long nij, long long nijH) {        // cut_bytes in 64 bits
        const long long yp = y_stride(nfp), qs = (nij * nk2) | 1, t = nij * s.nT * yp * 8, o = s.nO * qs * 16;
        return s.hs * nijH * nk2 * 16 + s.nE * qs * 16 + std::max(t, o) + s.NC * nfp * yp * 8;
    };
    const long long least = bytes(1, npp), most = bytes(npp, npp);
    for (int ti = 0; ti < 4; ++ti) {
        const long long room = (long long)tiers[ti].kb * 1024 - tables;
        p.threads = tiers[ti].threads;
        p.pool = (int)(std::min(std::max(most, 4096LL), room) / 16 * 16);
        if (least <= room) break;
    }
    return p;
}

int eri_default_threads(const EriShape &shape, bool gauge) {
    return eri_plan(shape.maxnfp, shape.maxLab, shape.maxnpp, gauge).threads;
}

namespace {
template <bool GAUGE, bool DF>
int resident_ctas(int threads, size_t smem) {
    int nb = 0, dev = 0, nsm = 0;
    QDT_CUDA_TRY(cudaGetDevice(&dev));
    QDT_CUDA_TRY(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
    QDT_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, eri_rows_kernel<GAUGE, DF>, threads, smem));
    return (nb > 0 ? nb : 1) * nsm;
}

template <bool GAUGE, bool DF>
void launch_rows(const EriParams *prms, const EriTask *tasks, int maxtasks, int *queue, const Plan &pl, int threads,
                 size_t smem, cudaStream_t s) {
    QDT_CUDA_TRY(cudaFuncSetAttribute(eri_rows_kernel<GAUGE, DF>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)smem));
    const int grid = min(maxtasks, resident_ctas<GAUGE, DF>(threads, smem));
    QDT_CUDA_TRY(cudaMemsetAsync(queue, 0, sizeof(int), s));
    eri_rows_kernel<GAUGE, DF><<<grid, threads, smem, s>>>(prms, tasks, queue, pl);
}
}  // namespace

void launch_eri(const EriParams *prms, const EriTask *tasks, int maxtasks, int *queue, const EriShape &shape,
                bool gauge, bool df, const EriLaunch &how, cudaStream_t s) {
    if (maxtasks <= 0) return;
    const Plan pl = eri_plan(shape.maxnfp, shape.maxLab, shape.maxnpp, gauge);
    const size_t smem = plan_smem(pl);
    const int threads = how.threads > 0 ? how.threads : pl.threads;
    if (threads % 32 || threads > 256) throw Error{QDT_ERR_ARG, "integral kernel: threads must be 32..256, a multiple of 32"};
    if (gauge) {
        if (df) launch_rows<true, true>(prms, tasks, maxtasks, queue, pl, threads, smem, s);
        else launch_rows<true, false>(prms, tasks, maxtasks, queue, pl, threads, smem, s);
    } else {
        if (df) launch_rows<false, true>(prms, tasks, maxtasks, queue, pl, threads, smem, s);
        else launch_rows<false, false>(prms, tasks, maxtasks, queue, pl, threads, smem, s);
    }
    QDT_CHECK_KERNEL("eri_rows_kernel");
}

// max over the entries of two integral-row blocks of |A - B| / (Q_row Q_col),
// rows and columns mapped to their shell pairs (mult 3: gauge rows (ab, I)).
__global__ void ratio_kernel(const double *A, const double *B, long long rows, long long ldw, int mult,
                             const int *row_pair, const int *col_pair, long long ncols, const double *Q,
                             double *out) {
    double m = 0.0;
    const long long total = rows * ldw;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total;
         e += (long long)gridDim.x * blockDim.x) {
        const long long r = e / ldw, c = e - r * ldw;
        if (c / mult >= ncols) continue;
        const double q = Q[row_pair[r / mult]] * Q[col_pair[c / mult]];
        const double d = fabs(A[e] - B[e]);
        if (d > 0.0) m = fmax(m, q > 0.0 ? d / q : INFINITY);
    }
    for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) atomicMax((unsigned long long *)out, (unsigned long long)__double_as_longlong(m));
}

void launch_ratio(const double *A, const double *B, long long rows, long long ldw, int mult, const int *row_pair,
                  const int *col_pair, long long ncols, const double *Q, double *out, cudaStream_t s) {
    if (rows <= 0 || ldw <= 0) return;
    long long blocks = std::min<long long>((rows * ldw + 255) / 256, 152 * 8);
    ratio_kernel<<<(unsigned)blocks, 256, 0, s>>>(A, B, rows, ldw, mult, row_pair, col_pair, ncols, Q, out);
    QDT_CHECK_LAUNCH();
}

void launch_split_pairs(const PairDev *pairs, int nsp, const double2 *E, long long n, float4 *E2, float2 *E1,
                        float2 *EX, cudaStream_t s) {
    if (n <= 0) return;
    bra_entries_kernel<<<nsp, 128, 0, s>>>(pairs, E, EX);
    QDT_CHECK_KERNEL("bra_entries_kernel");
    split_pairs_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(E, n, E2, E1);
    QDT_CHECK_KERNEL("split_pairs_kernel");
}

// Schwarz diagonals: Q[AB] = max over ab of sqrt(|(ab|ab)|), Coulomb kernel.
__global__ void __launch_bounds__(256, 2) schwarz_kernel(PairTables tb, const PairDev *pairs, Plan pl, double *Q) {
    const PairDev &AB = pairs[blockIdx.x];
    build_tables(pl);
    if (threadIdx.x == 0) tile_state().ket[0] = KetRef{AB.eoff, 0, 0, -1, AB.ppoff, (int)blockIdx.x, 0, 0};
    __syncthreads();
    set_tile(tb, AB, AB, false, false, 1, pl.pool);
    double qmax = 0.0;
    quartet_blocks<false, kF64>([&](const Group &g, auto value) {
        for (int x = threadIdx.x; x < g.xch; x += blockDim.x) {
            const int y = g.x0 + x - g.y0;
            if (y >= 0 && y < g.ych) qmax = fmax(qmax, sqrt(fabs(value(0, 0, x, y))));
        }
    });
    double *red = at_byte<double>(tile_state().o_pool);       // the block's last use of the pool is over
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) qmax = fmax(qmax, __shfl_xor_sync(0xffffffffu, qmax, o));
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = qmax;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < (int)(blockDim.x >> 5); ++w) qmax = fmax(qmax, red[w]);
        Q[blockIdx.x] = qmax;
    }
}

void launch_schwarz(const PairClass &pc, const double *boys, double *Q, cudaStream_t s) {
    if (pc.nsp <= 0) return;
    const Plan pl = eri_plan(pc.maxnfp, pc.maxLab, pc.maxnpp, false);
    const size_t smem = plan_smem(pl);
    QDT_CUDA_TRY(cudaFuncSetAttribute(schwarz_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    const PairTables tb{pc.d_pp, pc.d_E, nullptr, nullptr, nullptr, pc.d_fp, pc.d_ch, boys};
    schwarz_kernel<<<pc.nsp, pl.threads, smem, s>>>(tb, pc.d_pairs, pl, Q);
    QDT_CHECK_LAUNCH();
}

}  // namespace qdt
