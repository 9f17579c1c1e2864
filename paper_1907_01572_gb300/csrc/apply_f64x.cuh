// FP64 operator apply on the tensor pipe (large levels; see apply_impl.cuh for
// the operator and the native kernels).
//
// GB300 issues two FP64 operations per clock and SM, so the native FP64 apply
// is bound by its multiply-adds (7 ms for 13 M DOFs).  Here every contraction
// of the apply -- the twelve volume passes, the face-normal derivatives and the
// mortar interpolations and their transposes -- runs as an exact product of
// digits on the FP16 tensor pipe (the splitting of Ozaki, Ogita, Oishi and
// Rump, Numer. Algorithms 59, 2012, in fixed point):
//
// * A vector of values with a common exponent is held as 64-bit integers v,
//   |v| < 2^58, and split into six balanced digits, v = sum_i v_i 2^(10 (5-i)),
//   |v_i| <= 512.  An operator R, scaled by a power of two so that its rows'
//   absolute sums are at most 1, is split into R = 2^-9 sum_j R_j 2^(-10 j),
//   |R_j| <= 512 (tables built on the host).
// * The products v_i R_j of level l = i + j <= 6 are summed by
//   mma.sync.m16n8k16 (two digit pairs side by side in k for up to 8 operands):
//   the digits are FP16 integers, the sums stay below 2^22, so the FP32
//   accumulators -- started from 1.5 * 2^23, which leaves the sum as an integer
//   in their low bits -- are exact.  The levels are recombined with integer
//   multiply-adds.  A result is rounded to a unit of 2^-58 of the largest value
//   (what is dropped, l >= 7, is a thousandth of that), a thirtieth of what FP64
//   rounding loses on a value of that size; every pass renormalises, so the
//   digits always start at the largest value present.
// * Pointwise work (metric terms, fluxes, sums into y) stays in FP64.
//
// An element (or a mortar flux) whose values are not finite or lie outside
// 2^(+-800) takes the FP64 code below instead (x64_native_*).
//
// Measured (native FP64 -> this path): 61,440 hp elements, 13.2 M DOFs, 7055 ->
// 3650 us; 7,680 hp elements 1274 -> 554 us; 4,096 elements of p = 7 979 -> 336
// us, of p = 3 224 -> 164 us; 1,056 elements of the cubed sphere, p 4..8, 414 ->
// 270 us.  Rounding (additivity on integer data, relative): p = 1 2.2e-16 ->
// 1.6e-16, p = 3 2.7e-16 -> 1.9e-16, p = 8 3.4e-16 -> 2.1e-16, hp mesh 2.8e-16 ->
// 1.8e-16, cubed sphere 3.1e-16 -> 1.8e-16.  The element kernel is bound by
// latency (31 % issue at 16 warps per SM, n = 8) with the FP64 units at 54 %
// (metric terms, conversions, sums); its tensor pipe is at 9 %.
#pragma once
#include "apply_impl.cuh"
#include "f64x_tables.h"

namespace dg {
namespace apply_detail {

typedef long long i64;
typedef unsigned long long u64;

constexpr unsigned kMagic = 0x4B400000u;   // bits of 1.5 * 2^23

__device__ __forceinline__ void mma_k16(float (&d)[4], unsigned a0, unsigned a1, unsigned a2, unsigned a3, unsigned b0,
                                        unsigned b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
        "{%0, %1, %2, %3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void mma_k8(float (&d)[4], unsigned a0, unsigned a1, unsigned b0) {
    asm("mma.sync.aligned.m16n8k8.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5}, {%6}, {%0, %1, %2, %3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a0), "r"(a1), "r"(b0));
}

// Digits of the pair (p, q) at k = 2t, 2t + 1, as half2 words.
__device__ __forceinline__ void digits(i64 p, i64 q, unsigned (&d)[kX64Digits]) {
    constexpr i64 kBias = 512 * (1LL + (1LL << 10) + (1LL << 20) + (1LL << 30) + (1LL << 40) + (1LL << 50));
    const u64 a = (u64)(p + kBias), b = (u64)(q + kBias);   // in [0, 2^60): unsigned digits, 512 above the balanced ones
    const unsigned al = (unsigned)a, ah = (unsigned)(a >> 32), bl = (unsigned)b, bh = (unsigned)(b >> 32);
    const unsigned x[kX64Digits] = {ah >> 18, ah >> 8, __funnelshift_r(al, ah, 30), al >> 20, al >> 10, al};
    const unsigned y[kX64Digits] = {bh >> 18, bh >> 8, __funnelshift_r(bl, bh, 30), bl >> 20, bl >> 10, bl};
#pragma unroll
    for (int i = 0; i < kX64Digits; ++i) {
        const unsigned w = (__byte_perm(x[i], y[i], 0x5410) & 0x03ff03ffu) | 0x64006400u;   // 1024 + digit
        asm("add.f16x2 %0, %1, %2;" : "=r"(d[i]) : "r"(w), "r"(0xe600e600u));               // - 1536
    }
}

// The digits of a tile: rows g (h = 0) and g + 8 (h = 1), one or two groups of 8 operands.
template <int K>
struct Tile {
    static constexpr int KG = (K + 7) / 8;
    unsigned a[KG][kX64Digits][2];
    // ld(k): the integer at operand k of this lane's row (0 outside the row)
    template <int H, typename LD>
    __device__ __forceinline__ void fill(int t, LD ld) {
#pragma unroll
        for (int g = 0; g < KG; ++g) {
            unsigned d[kX64Digits];
            digits(ld(8 * g + 2 * t), ld(8 * g + 2 * t + 1), d);
#pragma unroll
            for (int i = 0; i < kX64Digits; ++i) a[g][i][H] = d[i];
        }
    }
    template <int H>
    __device__ __forceinline__ void clear() {
#pragma unroll
        for (int g = 0; g < KG; ++g)
#pragma unroll
            for (int i = 0; i < kX64Digits; ++i) a[g][i][H] = 0u;
    }
};

__device__ __forceinline__ void start(float (&d)[4]) {
#pragma unroll
    for (int i = 0; i < 4; ++i) d[i] = __uint_as_float(kMagic);
}

// acc += v_i R_j + v_i2 R_j2 (digit pairs of one level); i2 < 0: one pair.
template <int K>
__device__ __forceinline__ void pair_mma(float (&acc)[4], const Tile<K>& A, const unsigned (&b)[Tile<K>::KG][kX64Digits],
                                         int i, int j, int i2, int j2) {
    if constexpr (Tile<K>::KG == 1) {
        if (i2 >= 0) mma_k16(acc, A.a[0][i][0], A.a[0][i][1], A.a[0][i2][0], A.a[0][i2][1], b[0][j], b[0][j2]);
        else mma_k8(acc, A.a[0][i][0], A.a[0][i][1], b[0][j]);
    } else {
        mma_k16(acc, A.a[0][i][0], A.a[0][i][1], A.a[1][i][0], A.a[1][i][1], b[0][j], b[1][j]);
        if (i2 >= 0) mma_k16(acc, A.a[0][i2][0], A.a[0][i2][1], A.a[1][i2][0], A.a[1][i2][1], b[0][j2], b[1][j2]);
    }
}

// Product of a tile with columns 8 nt .. 8 nt + 7 of an operator (digit words W):
// o[2 h + c] = the value of row (h) and column 8 nt + 2 t + c, for the halves asked for.
template <int K, bool H0, bool H1>
__device__ __forceinline__ void tile_product(const Tile<K>& A, const unsigned* __restrict__ W, int nt, int lane,
                                             i64 (&o)[4]) {
    constexpr int KG = Tile<K>::KG;
    unsigned b[KG][kX64Digits];
#pragma unroll
    for (int g = 0; g < KG; ++g)
#pragma unroll
        for (int j = 0; j < kX64Digits; ++j) b[g][j] = W[((nt * KG + g) * kX64Digits + j) * 32 + lane];
    int t[4];
    {   // level 5, in units of 2^-9; level 6 joins it with the operator's digits scaled by 2^-10 (the
        // accumulators drop its fractions of a unit)
        unsigned c[KG][kX64Digits];
#pragma unroll
        for (int g = 0; g < KG; ++g)
#pragma unroll
            for (int j = 1; j < kX64Digits; ++j) asm("mul.f16x2 %0, %1, %2;" : "=r"(c[g][j]) : "r"(b[g][j]), "r"(0x14001400u));
        float p[4], q[4], r[4];
        start(p);
        start(q);
        start(r);
        pair_mma<K>(p, A, c, 1, 5, 2, 4);
        pair_mma<K>(q, A, c, 3, 3, 4, 2);
        pair_mma<K>(r, A, c, 5, 1, -1, -1);
        pair_mma<K>(p, A, b, 0, 5, 1, 4);
        pair_mma<K>(q, A, b, 2, 3, 3, 2);
        pair_mma<K>(r, A, b, 4, 1, 5, 0);
#pragma unroll
        for (int i = 0; i < 4; ++i)
            t[i] = (int)(__float_as_uint(p[i]) + __float_as_uint(q[i]) + __float_as_uint(r[i]) + (256u - 3u * kMagic)) >> 9;
    }
    {   // level 4, weight 2
        float p[4], q[4];
        start(p);
        start(q);
        pair_mma<K>(p, A, b, 0, 4, 1, 3);
        pair_mma<K>(q, A, b, 2, 2, 3, 1);
        pair_mma<K>(q, A, b, 4, 0, -1, -1);
#pragma unroll
        for (int i = 0; i < 4; ++i) t[i] += 2 * (int)(__float_as_uint(p[i]) + __float_as_uint(q[i]) - 2u * kMagic);
    }
    {   // level 3, weight 2^11
        float p[4], q[4];
        start(p);
        start(q);
        pair_mma<K>(p, A, b, 0, 3, 1, 2);
        pair_mma<K>(q, A, b, 2, 1, 3, 0);
#pragma unroll
        for (int i = 0; i < 4; ++i)
            o[i] = (i64)(int)(__float_as_uint(p[i]) + __float_as_uint(q[i]) - 2u * kMagic) * 2048 + t[i];
    }
    {   // level 2, weight 2^21
        float p[4];
        start(p);
        pair_mma<K>(p, A, b, 0, 2, 1, 1);
        pair_mma<K>(p, A, b, 2, 0, -1, -1);
#pragma unroll
        for (int i = 0; i < 4; ++i) o[i] += (i64)(int)(__float_as_uint(p[i]) - kMagic) * (1 << 21);
    }
    {   // levels 1 and 0, weights 2^31 and 2^41
        float p[4], q[4];
        start(p);
        start(q);
        pair_mma<K>(p, A, b, 0, 1, 1, 0);
        pair_mma<K>(q, A, b, 0, 0, -1, -1);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const unsigned c = __float_as_uint(p[i]) + (__float_as_uint(q[i]) << 10) - (kMagic + (kMagic << 10));
            o[i] += (i64)(int)(2u * c) * (1 << 30);
        }
    }
    (void)H0;
    (void)H1;
}

__device__ __forceinline__ unsigned abs_hi(i64 v) {
    const int h = (int)(v >> 32);
    return (unsigned)(h ^ (h >> 31));
}
// Left shift that brings values with the largest abs_hi m up to |v| < 2^58.
__device__ __forceinline__ int shift_of(unsigned m) { return max(__clz((int)m) - 6, 0); }
__device__ __forceinline__ int norm_shift(unsigned m) { return shift_of(__reduce_max_sync(0xffffffffu, m)); }

// Largest m of the CTA, in every thread; also a barrier.  Each call of an
// element uses a row of sh of its own.
template <int W>
__device__ __forceinline__ unsigned cta_max(unsigned m, unsigned (*sh)[W], int row) {
    m = __reduce_max_sync(0xffffffffu, m);
    if ((threadIdx.x & 31) == 0) sh[row][threadIdx.x >> 5] = m;
    __syncthreads();
#pragma unroll
    for (int w = 0; w < W; ++w) m = max(m, sh[row][w]);
    return m;
}
__device__ __forceinline__ i64 shr_round(i64 v, int s) {   // v / 2^s, s >= 0
    s = s > 62 ? 62 : s;
    return (v + ((1LL << s) >> 1)) >> s;
}

// Biased exponent of a value from its high word; the range in which every
// scaled quantity of the apply stays a normal FP64 number.
constexpr int kExpLo = 1023 - 800, kExpHi = 1023 + 800, kExpOff = 1080;
__device__ __forceinline__ bool exp_ok(int e) { return e >= kExpLo && e <= kExpHi; }
__device__ __forceinline__ unsigned abs_hi(double x) { return (unsigned)__double2hiint(x) & 0x7fffffffu; }

// round(x * 2^(1080 - eref)): |v| < 2^58 where x's exponent is at most eref.
__device__ __forceinline__ i64 to_fixed(double x, int eref) {
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
    const int ex = (int)((hi >> 20) & 0x7ff);
    const u64 m = ((u64)((hi & 0xfffffu) | (ex ? 0x100000u : 0u)) << 32 | lo) << 5;
    int d = eref - (ex ? ex : 1);
    d = d > 62 ? 62 : d;
    const i64 v = (i64)((m + ((1ull << d) >> 1)) >> d);
    return (int)hi < 0 ? -v : v;
}
// v * 2^e, correctly rounded (the result is a normal number: see exp_ok).
__device__ __forceinline__ double to_double(i64 v, int e) {
    const double x = (double)v;
    return v == 0 ? 0.0 : __hiloint2double(__double2hiint(x) + (e << 20), __double2loint(x));
}
__device__ __forceinline__ double scaled(double x, int e) {   // x * 2^e for a normal result, 0 for 0
    return (__double2hiint(x) & 0x7ff00000) == 0 ? 0.0 : __hiloint2double(__double2hiint(x) + (e << 20), __double2loint(x));
}

// One volume pass over the N^2 pencils along DIR: out (+)= R in, `in` read by
// ld(index) as normalised integers; returns the largest abs_hi of the results.
// The tiles of 16 pencils are dealt to the CTA's warps, from warp w on.
template <int N, int W, int DIR, bool ACC, typename LD>
__device__ __forceinline__ unsigned x64_pass(i64* __restrict__ out, const unsigned* __restrict__ op, int w, int lane,
                                             LD ld) {
    constexpr int stride = DIR == 0 ? 1 : (DIR == 1 ? Strides<N>::S1 : Strides<N>::S2);
    constexpr int NN = N * N, TILES = (NN + 15) / 16, NT = (N + 7) / 8;
    const int g = lane >> 2, t = lane & 3;
    unsigned mx = 0;
#pragma unroll 1
    for (int tile = w; tile < TILES; tile += W) {
        const int p0 = 16 * tile + g, p1 = p0 + 8;
        const bool v0 = p0 < NN, v1 = p1 < NN;
        const int b0 = pencil_base<N, DIR>(v0 ? p0 : 0), b1 = pencil_base<N, DIR>(v1 ? p1 : 0);
        Tile<N> A;
        A.template fill<0>(t, [&](int k) { return v0 && k < N ? ld(b0 + k * stride) : 0LL; });
        A.template fill<1>(t, [&](int k) { return v1 && k < N ? ld(b1 + k * stride) : 0LL; });
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
            i64 o[4];
            tile_product<N, true, true>(A, op, nt, lane, o);
#pragma unroll
            for (int h = 0; h < 2; ++h)
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    const int col = 8 * nt + 2 * t + c;
                    if ((h ? v1 : v0) && col < N) {
                        const int idx = (h ? b1 : b0) + col * stride;
                        const i64 v = ACC ? out[idx] + o[2 * h + c] : o[2 * h + c];
                        out[idx] = v;
                        mx = max(mx, abs_hi(v));
                    }
                }
        }
    }
    return mx;
}

// FP64 code for the elements and fluxes the integers cannot hold (run-time
// sizes, not inlined: it must not cost the kernels registers).
static __device__ __noinline__ void x64_native_pass(const double* in, double* out, const double* M, int n, int s1, int s2,
                                             int dir, bool trans, bool acc, int lane) {
    const int st[3] = {1, s1, s2};
    for (int k = lane; k < n * n * n; k += 32) {
        const int ix[3] = {k % n, (k / n) % n, k / (n * n)};
        const int o = ix[0] + s1 * ix[1] + s2 * ix[2], i = ix[dir], b = o - i * st[dir];
        double s = 0.0;
        for (int m = 0; m < n; ++m) s += (trans ? M[m * n + i] : M[i * n + m]) * in[b + m * st[dir]];
        out[o] = acc ? out[o] + s : s;
    }
    __syncwarp();
}

// Volume terms of one element in FP64 into Y (arrays as in element_body).
static __device__ __noinline__ void x64_native_volume(const double* x, const double* Ge, const double* c0e, const double* I,
                                               const double* Dg, double* Y, double* A, double* G1, double* U, int n,
                                               int s1, int s2, int lane) {
    const int n3 = n * n * n;
    auto at = [&](int k) { return k % n + s1 * ((k / n) % n) + s2 * (k / (n * n)); };
    for (int k = lane; k < n3; k += 32) U[at(k)] = x[k];
    __syncwarp();
    x64_native_pass(U, A, I, n, s1, s2, 0, false, false, lane);
    x64_native_pass(A, G1, I, n, s1, s2, 1, false, false, lane);
    x64_native_pass(G1, A, I, n, s1, s2, 2, false, false, lane);
    x64_native_pass(A, G1, Dg, n, s1, s2, 0, false, false, lane);
    x64_native_pass(A, Y, Dg, n, s1, s2, 1, false, false, lane);
    x64_native_pass(A, U, Dg, n, s1, s2, 2, false, false, lane);
    for (int k = lane; k < n3; k += 32) {
        const int s = at(k);
        const double g0 = G1[s], g1 = Y[s], g2 = U[s];
        const double m00 = Ge[k], m01 = Ge[n3 + k], m02 = Ge[2 * n3 + k], m11 = Ge[3 * n3 + k], m12 = Ge[4 * n3 + k],
                     m22 = Ge[5 * n3 + k];
        G1[s] = m00 * g0 + m01 * g1 + m02 * g2;
        Y[s] = m01 * g0 + m11 * g1 + m12 * g2;
        U[s] = m02 * g0 + m12 * g1 + m22 * g2;
        A[s] = c0e ? c0e[k] * A[s] : 0.0;
    }
    __syncwarp();
    x64_native_pass(G1, A, Dg, n, s1, s2, 0, true, true, lane);
    x64_native_pass(Y, A, Dg, n, s1, s2, 1, true, true, lane);
    x64_native_pass(U, A, Dg, n, s1, s2, 2, true, true, lane);
    x64_native_pass(A, G1, I, n, s1, s2, 0, true, false, lane);
    x64_native_pass(G1, U, I, n, s1, s2, 1, true, false, lane);
    x64_native_pass(U, Y, I, n, s1, s2, 2, true, false, lane);
}

// Trace of one mortar side in FP64 from the element's global values (trace_slot).
static __device__ __noinline__ void x64_native_trace(const double* x, int n, int q, int f, int o, const double* M1,
                                              const double* M2, const double* DL, const double* co, double* out,
                                              double* F, int lane) {
    const int n2 = n * n, q2 = q * q, d = f >> 1, fn = (f & 1) ? n - 1 : 0;
    int t1, t2;
    tangential(d, t1, t2);
    const int st[3] = {1, n, n2};
    double *uf = F, *df = uf + n2, *U1 = df + n2, *D1 = U1 + q * n, *N1 = D1 + q * n;
    for (int k = lane; k < n2; k += 32) {
        const int b = (k % n) * st[t1] + (k / n) * st[t2];
        double s = 0.0;
        for (int c = 0; c < n; ++c) s += DL[fn * n + c] * x[b + c * st[d]];
        uf[k] = x[b + fn * st[d]];
        df[k] = s;
    }
    __syncwarp();
    for (int k = lane; k < q * n; k += 32) {
        const int i1 = k % q, b = k / q;
        double su = 0, sd = 0, sn = 0;
        for (int a = 0; a < n; ++a) {
            const double iv = M1[2 * (i1 * n + a)], dv = M1[2 * (i1 * n + a) + 1];
            su += iv * uf[a + n * b];
            sd += dv * uf[a + n * b];
            sn += iv * df[a + n * b];
        }
        U1[k] = su;
        D1[k] = sd;
        N1[k] = sn;
    }
    __syncwarp();
    for (int k = lane; k < q2; k += 32) {
        const int i1 = k % q, i2 = k / q;
        int b1 = (o & 2) ? q - 1 - i1 : i1, b2 = (o & 4) ? q - 1 - i2 : i2;
        const int kA = (o & 1) ? b2 + q * b1 : b1 + q * b2;   // MortarMap
        double u = 0, g1 = 0, g2 = 0, gn = 0;
        for (int b = 0; b < n; ++b) {
            const double iv = M2[2 * (i2 * n + b)], dv = M2[2 * (i2 * n + b) + 1];
            u += iv * U1[i1 + q * b];
            g1 += iv * D1[i1 + q * b];
            g2 += dv * U1[i1 + q * b];
            gn += iv * N1[i1 + q * b];
        }
        out[kA] = u;
        out[q2 + kA] = co[t1 * q2 + kA] * g1 + co[t2 * q2 + kA] * g2 + co[d * q2 + kA] * gn;
    }
    __syncwarp();
}

// Lift of one mortar's flux factors P (PA, PB1, PB2, PBn) in FP64 (lift_apply) into the face's fu and fd.
static __device__ __noinline__ void x64_native_lift(const double* P, double* X, double* FU, double* FD, int n, int q,
                                                    const double* M1, const double* M2, int lane) {
    const int n2 = n * n, q2 = q * q;
    for (int k = lane; k < q * n; k += 32) {
        const int i1 = k % q, b = k / q;
        double a1 = 0, a2 = 0, a3 = 0;
        for (int i2 = 0; i2 < q; ++i2) {
            const double iv = M2[2 * (i2 * n + b)], dv = M2[2 * (i2 * n + b) + 1];
            const int p = i1 + q * i2;
            a1 += iv * P[p] + dv * P[2 * q2 + p];
            a2 += iv * P[q2 + p];
            a3 += iv * P[3 * q2 + p];
        }
        X[k] = a1;
        X[q * n + k] = a2;
        X[2 * q * n + k] = a3;
    }
    __syncwarp();
    for (int k = lane; k < n2; k += 32) {
        const int a = k % n, b = k / n;
        double fu = 0, fd = 0;
        for (int i1 = 0; i1 < q; ++i1) {
            const double iv = M1[2 * (i1 * n + a)], dv = M1[2 * (i1 * n + a) + 1];
            fu += iv * X[i1 + q * b] + dv * X[q * n + i1 + q * b];
            fd += iv * X[2 * q * n + i1 + q * b];
        }
        FU[k] += fu;
        FD[k] += fd;
    }
    __syncwarp();
}

// Exponent of the element's largest input value (v: this thread's values); false
// if the integers cannot hold the element.  A barrier.
template <int W, int R>
__device__ __forceinline__ bool element_exponent(const double (&v)[R], unsigned (*sh)[W], int row, int& eref) {
    unsigned m = 0;
#pragma unroll
    for (int j = 0; j < R; ++j) m = max(m, max(abs_hi(v[j]), __double2loint(v[j]) ? 1u : 0u));   // 1: a subnormal's low word
    m = cta_max(m, sh, row);
    eref = m == 0 ? 1023 : (int)(m >> 20);
    return exp_ok(eref);
}

// ---- trace kernel -------------------------------------------------------------------
// Shared memory of an element's CTA (in 8-byte values).
template <int N, int W>
struct X64Layout {
    static constexpr int NR = r4(Strides<N>::SIZE), OPW = x64_op_words(N, N) / 2;
    static constexpr int TTAB = OPW + r4(N * N);                    // DL ends' digits, DL
    static constexpr int TDF = 6 * N * N, TSCR = 3 * kQ * N;        // normal derivatives on the faces; per warp
    static constexpr int TSCRN = 2 * N * N + 3 * kQ * N;            // ... of the FP64 code (one warp)
    static constexpr int TSIZE = r4(TTAB + NR + TDF + (W * TSCR > TSCRN ? W * TSCR : TSCRN));
    static constexpr int ETAB = 4 * OPW + r4(N * N);
    static constexpr int ESCR = 4 * kQ * kQ + 3 * kQ * N;           // per warp: flux factors, lift
    // Y, then A, G1, U (dead after the volume terms) or the warps' scratch, then fu and fd of the six faces
    static constexpr int EBUF = 3 * NR > W * ESCR ? 3 * NR : W * ESCR;
    static constexpr int ESIZE = r4(ETAB + NR + EBUF + 12 * N * N);
};

// Digit words of mortar operator op (0 Im, 1 Dm, 2 Im^T, 3 Dm^T) of sides of N; QM = 9 for Q = 9, else 8
// (operators of up to 8 rows and operands all take the same words, so that Q can be a run-time value).
template <int N, int QM>
__device__ __forceinline__ const unsigned* x64_face_op(const unsigned* FW, int Q, int pos, int op) {
    constexpr int base = x64_face_off(N, N, 0, 0), per_q = 12 * x64_op_words(N, N), words = x64_op_words(QM, N);
    return FW + base + (Q - N) * per_q + (pos * 4 + op) * words;
}

// Point (j1, j2) of this side's face grid in the mortar's point order (MortarMap).
__device__ __forceinline__ int x64_point(int o, int Q, int j1, int j2) {
    const int b1 = (o & 2) ? Q - 1 - j1 : j1, b2 = (o & 4) ? Q - 1 - j2 : j2;
    return (o & 1) ? b2 + Q * b1 : b1 + Q * b2;
}

// Trace of this side at the Q x Q mortar points from the integers of the element (see trace_slot).
template <int N, int QM>
__device__ __forceinline__ void x64_trace_slot(const SlotInfo<double>& s, const i64* __restrict__ U,
                                               const i64* __restrict__ DF, int kd, int exU, int exD,
                                               const unsigned* __restrict__ FW, const int* __restrict__ FS, i64* X,
                                               const double* __restrict__ co, double* __restrict__ mt, int lane) {
    {
        constexpr int NTQ = (QM + 7) / 8, HN = (N + 7) / 8, HQ = (QM + 7) / 8;
        const int Q = s.q, Q2 = Q * Q;
        const int d = s.f >> 1, fn = (s.f & 1) ? N - 1 : 0, g = lane >> 2, t = lane & 3;
        int t1, t2;
        tangential(d, t1, t2);
        const int st1 = stride_of<N>(t1), st2 = stride_of<N>(t2), fo = fn * stride_of<N>(d);
        const i64* D = DF + (fn ? N * N : 0);
        const unsigned* I1 = x64_face_op<N, QM>(FW, Q, s.p0, 0);
        const unsigned* D1 = x64_face_op<N, QM>(FW, Q, s.p0, 1);
        const unsigned* I2 = x64_face_op<N, QM>(FW, Q, s.p1, 0);
        const unsigned* D2 = x64_face_op<N, QM>(FW, Q, s.p1, 1);
        const int sI = FS[x64_face_scale(N, Q)], sD = FS[x64_face_scale(N, Q) + 1];
        i64 *XU = X, *XD = XU + Q * N, *XN = XD + Q * N;   // [i1 + Q b]
        double cv[2][3] = {{0, 0, 0}, {0, 0, 0}};   // QM = 8: this lane's two points, loaded ahead of the passes
        if constexpr (QM == 8)
#pragma unroll
            for (int c = 0; c < 2; ++c)
                if (g < Q && 2 * t + c < Q) {
                    const int kA = x64_point(s.o, Q, g, 2 * t + c);
                    cv[c][0] = co[t1 * Q2 + kA];
                    cv[c][1] = co[t2 * Q2 + kA];
                    cv[c][2] = co[d * Q2 + kA];
                }
        unsigned mu = 0, md = 0, mn = 0;
#pragma unroll
        for (int hb = 0; hb < HN; ++hb) {
            const int b = 8 * hb + g;
            const bool v = b < N;
            Tile<N> A;
            A.template fill<0>(t, [&](int k) { return v && k < N ? U[k * st1 + b * st2 + fo] : 0LL; });
            A.template fill<1>(t, [&](int k) { return v && k < N ? D[k + N * b] << kd : 0LL; });
#pragma unroll
            for (int nt = 0; nt < NTQ; ++nt) {
                i64 o[4], e[4];
                tile_product<N, true, true>(A, I1, nt, lane, o);
                tile_product<N, true, false>(A, D1, nt, lane, e);
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    const int i1 = 8 * nt + 2 * t + c;
                    if (v && i1 < Q) {
                        XU[i1 + Q * b] = o[c];
                        XN[i1 + Q * b] = o[2 + c];
                        XD[i1 + Q * b] = e[c];
                        mu = max(mu, abs_hi(o[c]));
                        mn = max(mn, abs_hi(o[2 + c]));
                        md = max(md, abs_hi(e[c]));
                    }
                }
            }
        }
        __syncwarp();
        const int ku = norm_shift(mu), kx = norm_shift(md), kn = norm_shift(mn);
        const int eu = exU + sI - ku + sI, e2 = exU + sI - ku + sD;         // u, d/dt2 u
        const int e1 = exU + sD - kx + sI, en = exD - kd + sI - kn + sI;    // d/dt1 u, dn u
        double* out = mt + 4 * s.goff + 2 * s.side * Q2;
#pragma unroll
        for (int hq = 0; hq < HQ; ++hq) {
            const int i1 = 8 * hq + g;
            const bool v = i1 < Q;
            Tile<N> A, B;
            A.template fill<0>(t, [&](int k) { return v && k < N ? XU[i1 + Q * k] << ku : 0LL; });
            A.template fill<1>(t, [&](int k) { return v && k < N ? XD[i1 + Q * k] << kx : 0LL; });
            B.template fill<0>(t, [&](int k) { return v && k < N ? XN[i1 + Q * k] << kn : 0LL; });
            B.template clear<1>();
#pragma unroll
            for (int nt = 0; nt < NTQ; ++nt) {
                i64 o[4], e[4], w[4];
                tile_product<N, true, true>(A, I2, nt, lane, o);
                tile_product<N, true, false>(A, D2, nt, lane, e);
                tile_product<N, true, false>(B, I2, nt, lane, w);
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    const int i2 = 8 * nt + 2 * t + c;
                    if (v && i2 < Q) {
                        const int kA = x64_point(s.o, Q, i1, i2);
                        out[kA] = to_double(o[c], eu);
                        const double c1 = QM == 8 ? cv[c][0] : co[t1 * Q2 + kA], c2 = QM == 8 ? cv[c][1] : co[t2 * Q2 + kA],
                                     cn = QM == 8 ? cv[c][2] : co[d * Q2 + kA];
                        out[Q2 + kA] = c1 * to_double(o[2 + c], e1) + c2 * to_double(e[c], e2) + cn * to_double(w[c], en);
                    }
                }
            }
        }
        __syncwarp();
    }
}

// One CTA per element, elements blk, blk + nblk, ... of the bucket.
template <int N, int W>
__device__ __forceinline__ void x64_trace_body(const LevelView<double>& L, const ElemDesc* __restrict__ bdesc,
                                               int count, const double* __restrict__ x, int blk, int nblk) {
    using Ly = X64Layout<N, W>;
    constexpr int N3 = N * N * N, R = (N3 + (32 * W) - 1) / (32 * W), TILES = (N * N + 15) / 16;
    extern __shared__ __align__(16) double x64_smem[];
    __shared__ unsigned red[4][W];
    unsigned* sW = reinterpret_cast<unsigned*>(x64_smem);
    double* sDL = x64_smem + Ly::OPW;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
    for (int k = tid; k < x64_op_words(2, N); k += (32 * W)) sW[k] = L.x64.w[x64_vol_off(N, kX64Ends) + k];
    for (int k = tid; k < N * N; k += (32 * W)) sDL[k] = L.tab[tab_n(TabIndex::DL, N) + k];
    const int sE = L.x64.s[x64_vol_scale(N) + kX64Ends];
    i64* U = reinterpret_cast<i64*>(x64_smem + Ly::TTAB);
    i64* DF = U + Ly::NR;                        // [direction][face][N^2]
    i64* X = DF + Ly::TDF + warp * Ly::TSCR;
    for (int ei = blk; ei < count; ei += nblk) {
        const ElemDesc de = bdesc[ei];
        WarpSlots<double> ws;
        ws.load(L, de.s0, de.s1, lane);
        double v[R];
#pragma unroll
        for (int j = 0; j < R; ++j) v[j] = tid + (32 * W) * j < N3 ? x[de.dofo + tid + (32 * W) * j] : 0.0;
        if (warp == 0) ws.prefetch(L, lane, false);
        int eref;
        if (!element_exponent(v, red, 0, eref)) {   // (the barrier also separates the elements' use of shared memory)
            if (warp == 0)
                for (int si = ws.s0; si < ws.s1; ++si) {
                    const SlotInfo<double> s = unpack_rec(ws.get(si));
                    const double* ft = L.ftab + face_seg_off(N);
                    x64_native_trace(x + de.dofo, N, s.q, s.f, s.o, ft + face_tab_off(N, s.q, s.p0),
                                     ft + face_tab_off(N, s.q, s.p1), sDL,
                                     L.mg + 7 * s.goff + (s.side == 0 ? 1 : 4) * s.q * s.q,
                                     L.mt + 4 * s.goff + 2 * s.side * s.q * s.q, x64_smem + Ly::TTAB + Ly::NR + Ly::TDF,
                                     lane);
                }
            __syncthreads();
            continue;
        }
#pragma unroll
        for (int j = 0; j < R; ++j) {
            const int k = tid + (32 * W) * j;
            if (k < N3) U[sidx<N>(k)] = to_fixed(v[j], eref);
        }
        __syncthreads();
        // face-normal derivatives of the six faces: the tiles of the three directions dealt to the warps
        unsigned md[3] = {0, 0, 0};
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            int t1, t2;
            tangential(d, t1, t2);
            const int sd = stride_of<N>(d), st1 = stride_of<N>(t1), st2 = stride_of<N>(t2);
#pragma unroll 1
            for (int tile = (warp + d * TILES) % W; tile < TILES; tile += W) {
                const int p0 = 16 * tile + g, p1 = p0 + 8;
                const bool v0 = p0 < N * N, v1 = p1 < N * N;
                const int b0 = v0 ? (p0 % N) * st1 + (p0 / N) * st2 : 0, b1 = v1 ? (p1 % N) * st1 + (p1 / N) * st2 : 0;
                Tile<N> A;
                A.template fill<0>(t, [&](int k) { return v0 && k < N ? U[b0 + k * sd] : 0LL; });
                A.template fill<1>(t, [&](int k) { return v1 && k < N ? U[b1 + k * sd] : 0LL; });
                i64 o[4];
                tile_product<N, true, true>(A, sW, 0, lane, o);
                if (t == 0) {   // columns 0, 1: the two faces
                    i64* D = DF + 2 * d * N * N;
#pragma unroll
                    for (int c = 0; c < 2; ++c) {
                        if (v0) D[c * N * N + p0] = o[c];
                        if (v1) D[c * N * N + p1] = o[2 + c];
                        if (v0) md[d] = max(md[d], abs_hi(o[c]));
                        if (v1) md[d] = max(md[d], abs_hi(o[2 + c]));
                    }
                }
            }
        }
        const int kd0 = shift_of(cta_max(md[0], red, 1)), kd1 = shift_of(cta_max(md[1], red, 2)),
                  kd2 = shift_of(cta_max(md[2], red, 3));
        const int exU = eref - kExpOff;
        for (int si = ws.s0 + warp; si < ws.s1; si += W) {
            const SlotInfo<double> s = unpack_rec(ws.get(si));
            const int d = s.f >> 1, kd = d == 0 ? kd0 : (d == 1 ? kd1 : kd2);
            const double* co = L.mg + 7 * s.goff + (s.side == 0 ? 1 : 4) * s.q * s.q;
            const i64* D = DF + 2 * d * N * N;
            if (N <= 8 && s.q <= 8)
                x64_trace_slot<N, (N > 8 ? 9 : 8)>(s, U, D, kd, exU, exU + sE, L.x64.w, L.x64.s, X, co, L.mt, lane);
            else
                x64_trace_slot<N, 9>(s, U, D, kd, exU, exU + sE, L.x64.w, L.x64.s, X, co, L.mt, lane);
        }
    }
}

// ---- element kernel -----------------------------------------------------------------
template <int N, int QM>
__device__ __forceinline__ void x64_lift_slot(const LevelView<double>& L, const SlotInfo<double>& s, bool interior,
                                              bool first, double sig, double* __restrict__ FU,
                                              double* __restrict__ FD,
                                              const unsigned* __restrict__ FW, const int* __restrict__ FS, double* F,
                                              const double* __restrict__ wSp, const double* __restrict__ co,
                                              const double* __restrict__ m, int lane) {
    {
        constexpr int NTN = (N + 7) / 8, HN = (N + 7) / 8, HQ = (QM + 7) / 8;
        const int Q = s.q, Q2 = Q * Q;
        const int d = s.f >> 1, g = lane >> 2, t = lane & 3;
        int t1, t2;
        tangential(d, t1, t2);
        double *PA = F, *P1 = PA + Q2, *P2 = P1 + Q2, *Pn = P2 + Q2;
        const double half = interior ? 0.5 : 1.0;
        // flux factors at a mortar point: pa, and b c_t1, b c_t2, b c_d
        auto flux = [&](int j1, int j2, double (&p)[4]) {
            const int kA = x64_point(s.o, Q, j1, j2);
            const double wS = wSp[kA], wh = half * wS;
            double j = m[kA], a = m[Q2 + kA];
            if (interior) {
                j -= m[2 * Q2 + kA];
                a += m[3 * Q2 + kA];
            }
            const double pa = sig * (wS * j) - wh * a, b = -(wh * j);
            p[0] = s.side == 0 ? pa : -pa;
            p[1] = b * co[t1 * Q2 + kA];
            p[2] = b * co[t2 * Q2 + kA];
            p[3] = b * co[d * Q2 + kA];
        };
        unsigned ma = 0, mb = 0;
        // QM = 8: a lane needs the fluxes of two points only, (g, 2t) and (g, 2t + 1), and keeps them in registers
        double pv[2][4] = {{0, 0, 0, 0}, {0, 0, 0, 0}};
        if constexpr (QM == 8) {
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                if (g < Q && 2 * t + c < Q) flux(g, 2 * t + c, pv[c]);
                ma = max(ma, abs_hi(pv[c][0]));
                mb = max(mb, max(abs_hi(pv[c][1]), max(abs_hi(pv[c][2]), abs_hi(pv[c][3]))));
            }
        } else {
            for (int k = lane; k < Q2; k += 32) {
                double p[4];
                flux(k % Q, k / Q, p);
                PA[k] = p[0];
                P1[k] = p[1];
                P2[k] = p[2];
                Pn[k] = p[3];
                ma = max(ma, abs_hi(p[0]));
                mb = max(mb, max(abs_hi(p[1]), max(abs_hi(p[2]), abs_hi(p[3]))));
            }
            __syncwarp();
        }
        ma = __reduce_max_sync(0xffffffffu, ma);
        mb = __reduce_max_sync(0xffffffffu, mb);
        int eA = (int)(ma >> 20), eB = (int)(mb >> 20);
        double* Xd = F + 4 * Q2;
        if ((ma != 0 && !exp_ok(eA)) || (mb != 0 && !exp_ok(eB))) {
            const double* ft = L.ftab + face_seg_off(N);
            if constexpr (QM == 8)
#pragma unroll
                for (int c = 0; c < 2; ++c)
                    if (g < Q && 2 * t + c < Q)
#pragma unroll
                        for (int i = 0; i < 4; ++i) F[i * Q2 + g + Q * (2 * t + c)] = pv[c][i];
            if (first)
                for (int k = lane; k < N * N; k += 32) FU[k] = FD[k] = 0.0;
            __syncwarp();
            x64_native_lift(PA, Xd, FU, FD, N, Q, ft + face_tab_off(N, Q, s.p0), ft + face_tab_off(N, Q, s.p1), lane);
            return;
        }
        if (ma == 0 && mb == 0) {   // (a flux below the smallest normal number counts as zero)
            if (first)
                for (int k = lane; k < N * N; k += 32) FU[k] = FD[k] = 0.0;
            return;
        }
        if (ma == 0) eA = eB;
        if (mb == 0) eB = eA;
        const unsigned* I1 = x64_face_op<N, QM>(FW, Q, s.p0, 2);
        const unsigned* D1 = x64_face_op<N, QM>(FW, Q, s.p0, 3);
        const unsigned* I2 = x64_face_op<N, QM>(FW, Q, s.p1, 2);
        const unsigned* D2 = x64_face_op<N, QM>(FW, Q, s.p1, 3);
        const int sI = FS[x64_face_scale(N, Q) + 2], sD = FS[x64_face_scale(N, Q) + 3];
        i64* X1 = reinterpret_cast<i64*>(Xd);   // [i1 + Q b]
        i64 *X2 = X1 + Q * N, *X3 = X2 + Q * N;
        const int exA = eA - kExpOff + sI, exB = eB - kExpOff + sI, exD = eB - kExpOff + sD;
        const int ex1 = max(exA, exD) + 1;      // X1 = I^T PA + D^T P2
        unsigned m1 = 0, m2 = 0, m3 = 0;
#pragma unroll
        for (int hq = 0; hq < HQ; ++hq) {
            const int i1 = 8 * hq + g;
            const bool v = i1 < Q;
            Tile<QM> A, B;
            auto at = [&](const double* P, int i, int k) { return QM == 8 ? pv[k & 1][i] : (v && k < Q ? P[i1 + Q * k] : 0.0); };
            A.template fill<0>(t, [&](int k) { return to_fixed(at(PA, 0, k), eA); });
            A.template fill<1>(t, [&](int k) { return to_fixed(at(P1, 1, k), eB); });
            B.template fill<0>(t, [&](int k) { return to_fixed(at(Pn, 3, k), eB); });
            B.template fill<1>(t, [&](int k) { return to_fixed(at(P2, 2, k), eB); });
#pragma unroll
            for (int nt = 0; nt < NTN; ++nt) {
                i64 o[4], w[4], e[4];
                tile_product<QM, true, true>(A, I2, nt, lane, o);
                tile_product<QM, true, false>(B, I2, nt, lane, w);
                tile_product<QM, false, true>(B, D2, nt, lane, e);
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    const int b = 8 * nt + 2 * t + c;
                    if (v && b < N) {
                        const i64 x1 = shr_round(o[c], ex1 - exA) + shr_round(e[2 + c], ex1 - exD);
                        X1[i1 + Q * b] = x1;
                        X2[i1 + Q * b] = o[2 + c];
                        X3[i1 + Q * b] = w[c];
                        m1 = max(m1, abs_hi(x1));
                        m2 = max(m2, abs_hi(o[2 + c]));
                        m3 = max(m3, abs_hi(w[c]));
                    }
                }
            }
        }
        __syncwarp();
        const int k1 = norm_shift(m1), k2 = norm_shift(m2), k3 = norm_shift(m3);
        const int e1 = ex1 - k1 + sI, e2 = exB - k2 + sD, e3 = exB - k3 + sI;
#pragma unroll
        for (int hb = 0; hb < HN; ++hb) {
            const int b = 8 * hb + g;
            const bool v = b < N;
            Tile<QM> A, B;
            A.template fill<0>(t, [&](int k) { return v && k < Q ? X1[k + Q * b] << k1 : 0LL; });
            A.template fill<1>(t, [&](int k) { return v && k < Q ? X3[k + Q * b] << k3 : 0LL; });
            B.template fill<0>(t, [&](int k) { return v && k < Q ? X2[k + Q * b] << k2 : 0LL; });
            B.template clear<1>();
#pragma unroll
            for (int nt = 0; nt < NTN; ++nt) {
                i64 o[4], w[4];
                tile_product<QM, true, true>(A, I1, nt, lane, o);
                tile_product<QM, true, false>(B, D1, nt, lane, w);
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    const int a = 8 * nt + 2 * t + c;
                    if (v && a < N) {
                        const double fu = to_double(o[c], e1) + to_double(w[c], e2), fd = to_double(o[2 + c], e3);
                        FU[a + N * b] = first ? fu : FU[a + N * b] + fu;
                        FD[a + N * b] = first ? fd : FD[a + N * b] + fd;
                    }
                }
            }
        }
        __syncwarp();
    }
}

// Volume terms of one element into Y, by the whole CTA; false (nothing in Y) if the integers cannot hold a
// quantity.  Ends with a barrier.
template <int N, int W>
__device__ __forceinline__ bool x64_volume(const double* __restrict__ x, const double* __restrict__ Ge,
                                           const double* __restrict__ c0e, const unsigned* sW, int sI, int sIT, int sD,
                                           int sDT, double* Yd, double* Ad, double* G1d, double* Ud,
                                           unsigned (*red)[W]) {
    constexpr int N3 = N * N * N, R = (N3 + (32 * W) - 1) / (32 * W), OPW = x64_op_words(N, N),
                  TILES = (N * N + 15) / 16;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    i64 *Y = reinterpret_cast<i64*>(Yd), *A = reinterpret_cast<i64*>(Ad), *G1 = reinterpret_cast<i64*>(G1d),
        *U = reinterpret_cast<i64*>(Ud);
    const unsigned *wI = sW, *wIT = wI + OPW, *wD = wIT + OPW, *wDT = wD + OPW;
    int eref;
    {
        double v[R];
#pragma unroll
        for (int j = 0; j < R; ++j) v[j] = tid + (32 * W) * j < N3 ? x[tid + (32 * W) * j] : 0.0;
        prefetch_l2(Ge, 6 * N3, tid, (32 * W));   // metric terms, needed after 6 passes
        if (!element_exponent(v, red, 0, eref)) return false;
#pragma unroll
        for (int j = 0; j < R; ++j) {
            const int k = tid + (32 * W) * j;
            if (k < N3) U[sidx<N>(k)] = to_fixed(v[j], eref);
        }
    }
    __syncthreads();
    unsigned mx = x64_pass<N, W, 0, false>(A, wI, warp, lane, [&](int i) { return U[i]; });
    const int k1 = shift_of(cta_max(mx, red, 1));
    mx = x64_pass<N, W, 1, false>(G1, wI, warp, lane, [&](int i) { return A[i] << k1; });
    const int k2 = shift_of(cta_max(mx, red, 2));
    mx = x64_pass<N, W, 2, false>(A, wI, warp, lane, [&](int i) { return G1[i] << k2; });
    const int k3 = shift_of(cta_max(mx, red, 3));
    const int exg = eref - kExpOff + 3 * sI - k1 - k2 - k3 + sD;   // exponent of the gradient's integers
    x64_pass<N, W, 0, false>(G1, wD, warp, lane, [&](int i) { return A[i] << k3; });
    x64_pass<N, W, 1, false>(Y, wD, (warp + TILES) % W, lane, [&](int i) { return A[i] << k3; });
    x64_pass<N, W, 2, false>(U, wD, (warp + 2 * TILES) % W, lane, [&](int i) { return A[i] << k3; });
    __syncthreads();
    unsigned mf = 0;
    for (int k = tid; k < N3; k += (32 * W)) {
        const int s = sidx<N>(k);
        const double m00 = __ldcs(Ge + k), m01 = __ldcs(Ge + N3 + k), m02 = __ldcs(Ge + 2 * N3 + k);
        const double m11 = __ldcs(Ge + 3 * N3 + k), m12 = __ldcs(Ge + 4 * N3 + k), m22 = __ldcs(Ge + 5 * N3 + k);
        const double g0 = (double)G1[s], g1 = (double)Y[s], g2 = (double)U[s];
        const double f0 = m00 * g0 + m01 * g1 + m02 * g2, f1 = m01 * g0 + m11 * g1 + m12 * g2,
                     f2 = m02 * g0 + m12 * g1 + m22 * g2;
        G1d[s] = f0;
        Yd[s] = f1;
        Ud[s] = f2;
        mf = max(mf, max(abs_hi(f0), max(abs_hi(f1), abs_hi(f2))));
        if (c0e) {   // c0 u in the units of the divergence's integers (see below)
            const double c = scaled(c0e[k] * (double)A[s], k3 - sD - sDT);
            Ad[s] = c;
            mf = max(mf, abs_hi(c));
        }
    }
    mf = cta_max(mf, red, 4);
    const int ef = mf == 0 ? 1023 : (int)(mf >> 20);
    // the fluxes' integers keep two spare bits, for the sum of three directions and the zeroth-order term
    const int er = ef + 2, exA = er - kExpOff + exg + sDT;
    if (!exp_ok(ef) || exA < -900 || exA > 800) return false;
    if (c0e) {
        for (int k = tid; k < N3; k += (32 * W)) A[sidx<N>(k)] = to_fixed(Ad[sidx<N>(k)], er);
        __syncthreads();
        x64_pass<N, W, 0, true>(A, wDT, warp, lane, [&](int i) { return to_fixed(G1d[i], er); });
    } else {
        x64_pass<N, W, 0, false>(A, wDT, warp, lane, [&](int i) { return to_fixed(G1d[i], er); });
    }
    __syncthreads();
    x64_pass<N, W, 1, true>(A, wDT, warp, lane, [&](int i) { return to_fixed(Yd[i], er); });
    __syncthreads();
    mx = x64_pass<N, W, 2, true>(A, wDT, warp, lane, [&](int i) { return to_fixed(Ud[i], er); });
    const int k4 = shift_of(cta_max(mx, red, 5));
    mx = x64_pass<N, W, 0, false>(G1, wIT, warp, lane, [&](int i) { return A[i] << k4; });
    const int k5 = shift_of(cta_max(mx, red, 6));
    mx = x64_pass<N, W, 1, false>(U, wIT, warp, lane, [&](int i) { return G1[i] << k5; });
    const int k6 = shift_of(cta_max(mx, red, 7));
    x64_pass<N, W, 2, false>(Y, wIT, warp, lane, [&](int i) { return U[i] << k6; });
    __syncthreads();
    const int ey = exA + 3 * sIT - k4 - k5 - k6;
    for (int k = tid; k < N3; k += (32 * W)) Yd[sidx<N>(k)] = to_double(Y[sidx<N>(k)], ey);
    __syncthreads();
    return true;
}

// Degrees whose volume terms stay in FP64: a pass of the integers takes the
// time of a tile (about 1.5 us of latency) however few pencils it has, and
// 12 n^4 FP64 multiply-adds are fewer than that up to n = 5.
template <int N>
constexpr bool x64_small() {
    return N <= 5;
}

template <int N, int W, int DIR, bool TRANS, bool ACC>
__device__ __forceinline__ void x64_small_pass(const double* __restrict__ in, double* __restrict__ out,
                                               const double* __restrict__ M) {
    constexpr int st = DIR == 0 ? 1 : (DIR == 1 ? Strides<N>::S1 : Strides<N>::S2);
#pragma unroll
    for (int k0 = 0; k0 < N * N * N; k0 += 32 * W) {
        const int k = k0 + threadIdx.x;
        if (k >= N * N * N) continue;
        const int i = DIR == 0 ? k % N : (DIR == 1 ? (k / N) % N : k / (N * N)), o = sidx<N>(k), b = o - i * st;
        double s = ACC ? out[o] : 0.0;
#pragma unroll
        for (int m = 0; m < N; ++m) s += (TRANS ? M[m * N + i] : M[i * N + m]) * in[b + m * st];
        out[o] = s;
    }
}

// Volume terms of one element into Y in FP64, by the whole CTA.  Ends with a barrier.
template <int N, int W>
__device__ __forceinline__ void x64_small_volume(const double* __restrict__ x, const double* __restrict__ Ge,
                                                 const double* __restrict__ c0e, const double* I, const double* D,
                                                 double* Y, double* A, double* G1, double* U) {
    constexpr int N3 = N * N * N;
    for (int k = threadIdx.x; k < N3; k += 32 * W) U[sidx<N>(k)] = x[k];
    prefetch_l2(Ge, 6 * N3, threadIdx.x, 32 * W);
    __syncthreads();
    x64_small_pass<N, W, 0, false, false>(U, A, I);
    __syncthreads();
    x64_small_pass<N, W, 1, false, false>(A, G1, I);
    __syncthreads();
    x64_small_pass<N, W, 2, false, false>(G1, A, I);
    __syncthreads();
    x64_small_pass<N, W, 0, false, false>(A, G1, D);
    x64_small_pass<N, W, 1, false, false>(A, Y, D);
    x64_small_pass<N, W, 2, false, false>(A, U, D);
    __syncthreads();
    for (int k = threadIdx.x; k < N3; k += 32 * W) {
        const int s = sidx<N>(k);
        const double m00 = __ldcs(Ge + k), m01 = __ldcs(Ge + N3 + k), m02 = __ldcs(Ge + 2 * N3 + k);
        const double m11 = __ldcs(Ge + 3 * N3 + k), m12 = __ldcs(Ge + 4 * N3 + k), m22 = __ldcs(Ge + 5 * N3 + k);
        const double g0 = G1[s], g1 = Y[s], g2 = U[s];
        G1[s] = m00 * g0 + m01 * g1 + m02 * g2;
        Y[s] = m01 * g0 + m11 * g1 + m12 * g2;
        U[s] = m02 * g0 + m12 * g1 + m22 * g2;
        A[s] = c0e ? c0e[k] * A[s] : 0.0;
    }
    __syncthreads();
    x64_small_pass<N, W, 0, true, true>(G1, A, D);
    __syncthreads();
    x64_small_pass<N, W, 1, true, true>(Y, A, D);
    __syncthreads();
    x64_small_pass<N, W, 2, true, true>(U, A, D);
    __syncthreads();
    x64_small_pass<N, W, 0, true, false>(A, G1, I);
    __syncthreads();
    x64_small_pass<N, W, 1, true, false>(G1, U, I);
    __syncthreads();
    x64_small_pass<N, W, 2, true, false>(U, Y, I);
    __syncthreads();
}

// One CTA per element: the volume passes' tiles are dealt to its warps, the
// faces too (each face into its own fu and fd, in slot order), and the nodes
// gather volume and face parts at the end.
template <int N, int W>
__device__ __forceinline__ void x64_element_body(const LevelView<double>& L, const ElemDesc* __restrict__ bdesc,
                                                 int count, const double* __restrict__ x, double* __restrict__ y,
                                                 int blk, int nblk) {
    using Ly = X64Layout<N, W>;
    constexpr int N2 = N * N, N3 = N2 * N, NR = Ly::NR, OPW = x64_op_words(N, N);
    extern __shared__ __align__(16) double x64_smem[];
    __shared__ unsigned red[8][W];
    unsigned* sW = reinterpret_cast<unsigned*>(x64_smem);
    double* sDL = x64_smem + 4 * Ly::OPW;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if constexpr (x64_small<N>()) {   // I and Dg themselves, in the place of their digits
        for (int k = tid; k < N2; k += (32 * W)) {
            x64_smem[k] = L.tab[tab_n(TabIndex::I, N) + k];
            x64_smem[N2 + k] = L.tab[tab_n(TabIndex::Dg, N) + k];
        }
        __syncthreads();
    } else {
        for (int k = tid; k < 4 * OPW; k += (32 * W)) sW[k] = L.x64.w[x64_vol_off(N, 0) + k];
    }
    for (int k = tid; k < N2; k += (32 * W)) sDL[k] = L.tab[tab_n(TabIndex::DL, N) + k];
    const int* vs = L.x64.s + x64_vol_scale(N);
    const int sI = vs[kX64I], sIT = vs[kX64IT], sD = vs[kX64D], sDT = vs[kX64DT];
    double* Y = x64_smem + Ly::ETAB;
    double *A = Y + NR, *G1 = A + NR, *U = G1 + NR, *F = A + warp * Ly::ESCR;
    double* FU = Y + NR + Ly::EBUF;      // [face][N^2]
    double* FD = FU + 6 * N2;
    for (int ei = blk; ei < count; ei += nblk) {
        const ElemDesc de = bdesc[ei];
        WarpSlots<double> ws;
        ws.load(L, de.s0, de.s1, lane);
        const double* Ge = L.G + 6 * de.vo;
        const double* c0e = L.c0 ? L.c0 + de.vo : nullptr;
        if (warp == 0) ws.prefetch(L, lane, true);
        if constexpr (x64_small<N>()) {
            x64_small_volume<N, W>(x + de.dofo, Ge, c0e, x64_smem, x64_smem + N2, Y, A, G1, U);
        } else if (!x64_volume<N, W>(x + de.dofo, Ge, c0e, sW, sI, sIT, sD, sDT, Y, A, G1, U, red)) {
            __syncthreads();
            if (warp == 0)
                x64_native_volume(x + de.dofo, Ge, c0e, L.tab + tab_n(TabIndex::I, N), L.tab + tab_n(TabIndex::Dg, N), Y,
                                  A, G1, U, N, Strides<N>::S1, Strides<N>::S2, lane);
            __syncthreads();
        }
        int face = -1;
        for (int si = ws.s0; si < ws.s1; ++si) {
            const SlotRec<double> r = ws.get(si);
            const SlotInfo<double> s = unpack_rec(r);
            if (s.f % W != warp) continue;
            const bool first = s.f != face;   // of its face: stores, the others add
            face = s.f;
            const bool interior = (r.info >> 12) & 1;
            const double* mg = L.mg + 7 * s.goff;
            const double* co = mg + (s.side == 0 ? 1 : 4) * s.q * s.q;
            const double* mt = L.mt + 4 * s.goff;
            double *fu = FU + s.f * N2, *fd = FD + s.f * N2;
            if (N <= 8 && s.q <= 8)
                x64_lift_slot<N, (N > 8 ? 9 : 8)>(L, s, interior, first, r.sig, fu, fd, L.x64.w, L.x64.s, F, mg, co, mt, lane);
            else
                x64_lift_slot<N, 9>(L, s, interior, first, r.sig, fu, fd, L.x64.w, L.x64.s, F, mg, co, mt, lane);
            __syncwarp();
        }
        __syncthreads();
        for (int k = tid; k < N3; k += (32 * W)) {
            const int c[3] = {k % N, (k / N) % N, k / N2};
            double v = Y[sidx<N>(k)];
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                const int i = (d == 0 ? c[1] : c[0]) + N * (d == 2 ? c[1] : c[2]);
                const double *fu = FU + 2 * d * N2 + i, *fd = FD + 2 * d * N2 + i;
                v += sDL[c[d]] * fd[0] + sDL[(N - 1) * N + c[d]] * fd[N2];
                if (c[d] == 0) v += fu[0];
                if (c[d] == N - 1) v += fu[N2];
            }
            if (L.Ob != nullptr) v += y[de.dofo + k];   // the Galerkin blocks' part (galerkin_apply_kernel)
            __stcs(y + de.dofo + k, v);
        }
        __syncthreads();
    }
}

// Warps of an element's CTA: two where there are elements enough to fill the
// chip (a pass has 1 to 6 tiles, an element six faces), four where the time of
// one element counts.
constexpr int kX64Warps = 2, kX64FusedWarps = 4;

template <int N>
__global__ void __launch_bounds__(32 * kX64Warps, (N > 8 ? 6 : 8))
    x64_trace_kernel(LevelView<double> L, const ElemDesc* __restrict__ bdesc, int count, const double* __restrict__ x) {
    x64_trace_body<N, kX64Warps>(L, bdesc, count, x, blockIdx.x, gridDim.x);
}
template <int N>
__global__ void __launch_bounds__(32 * kX64Warps, (N > 8 ? 6 : 8))
    x64_element_kernel(LevelView<double> L, const ElemDesc* __restrict__ bdesc, int count, const double* __restrict__ x,
                       double* __restrict__ y) {
    x64_element_body<N, kX64Warps>(L, bdesc, count, x, y, blockIdx.x, gridDim.x);
}

// Launches of one degree (apply_f64x_launch.cuh, instantiated in apply_f64x_a.cu to apply_f64x_d.cu).
template <int N>
cudaError_t launch_x64_trace(const LevelView<double>& L, const BucketInfo& b, const double* x, cudaStream_t st);
template <int N>
cudaError_t launch_x64_element(const LevelView<double>& L, const BucketInfo& b, const double* x, double* y,
                               cudaStream_t st);

}  // namespace apply_detail
}  // namespace dg
