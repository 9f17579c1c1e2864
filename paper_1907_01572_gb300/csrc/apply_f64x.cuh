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
// * The operands of one contraction (a pencil, a row of a face's points) share an
//   exponent, that of the largest of them: they are held as integers v, |v| <=
//   2^58, and split into six balanced digits, v = sum_i v_i 2^(10 (5-i)),
//   |v_i| <= 512.  An operator R, scaled by a power of two so that its rows'
//   absolute sums are at most 1, is split into R = 2^-9 sum_j R_j 2^(-10 j),
//   |R_j| <= 512 (tables built on the host).
// * The products v_i R_j of level l = i + j <= 6 are summed by
//   mma.sync.m16n8k16 (two digit pairs side by side in k for up to 8 operands):
//   the digits are FP16 integers, the sums stay below 2^22, so the FP32
//   accumulators -- started from 1.5 * 2^23, which leaves the sum as an integer
//   in their low bits -- are exact.  The levels are recombined with integer
//   multiply-adds.  A result is rounded to 2^-58 of its own pencil's largest
//   operand (what is dropped, l >= 7, is a thousandth of that).
// * Between the volume passes values are FP64 numbers, so every pencil of the
//   next direction takes the exponent of its own values; between the two passes
//   of a face they stay integers with the exponents of the rows that wrote them,
//   and are brought to the exponent of their new row as they are read.
// * Pointwise work (metric terms, fluxes, sums into y) stays in FP64.
//
// Accuracy: a result is off by 2^-58 of its pencil's largest operand times the
// scale of R, and (volume) by its own rounding to FP64; FP64 multiply-adds are off
// by 2^-53 of every term.  So the digits lose on an entry only where a pencil's
// values or R's entries span more than about 2^5 and the small ones alone make
// the result.  (One exponent for a whole element, which this replaced, lost 5 to
// 12 times FP64's error in norm, and 100 times at small entries, on values that
// are concentrated in a part of the element.)  Relative error of the volume term
// of one affine element against 200-bit arithmetic, FP64 -> digits, 2-norm (and
// median entry), n = 8: N(0, 1) 3.1e-16 -> 1.8e-16 (2.8e-16 -> 1.8e-16); 1 at a
// corner node 1.0e-15 -> 3.8e-16 (5.5e-16 -> 4.6e-16); r^-5 with the centre 0.2
// off a corner 1.8e-15 -> 5.9e-16 (3.4e-15 -> 3.7e-15); exp(-30 (x + y + z))
// 8.7e-16 -> 4.3e-16 (6.4e-16 -> 5.7e-16); magnitudes over 10^8 at random 3.4e-16
// -> 1.8e-16 (4.4e-16 -> 2.5e-16).  Whole apply (additivity on integer data): p = 1
// 2.2e-16 -> 1.6e-16, p = 3 2.7e-16 -> 1.9e-16, p = 8 3.4e-16 -> 2.0e-16, hp mesh
// 2.8e-16 -> 1.7e-16, cubed sphere 3.1e-16 -> 1.7e-16.
//
// A pencil whose values are not finite or have none between 2^-800 and 2^801
// takes FP64 code instead (x64_native_*), a mortar with such a row whole.
//
// Measured (native FP64 -> this path): 61,440 hp elements, 13.2 M DOFs, 7055 ->
// 4200 us; 7,680 hp elements 1274 -> 560..650 us; 4,096 elements of p = 7 979 ->
// 374 us, of p = 3 224 -> 174 us; 1,056 elements of the cubed sphere, p 4..8, 414
// -> 300 us.  The exponent per pencil costs 15 to 20 % of that (one per element:
// 3642, 549, 335, 163 and 267 us): the largest of eight values over four lanes
// and the conversions.  A conversion of 64-bit integers takes a warp 64 clocks of
// its quarter's FP64 unit, the element kernel's fullest: in the faces the
// integers are kept (4,096 elements of p = 3: 192 -> 175 us), in the passes of n
// <= 8 they are converted in integer instructions (p = 7: 401 -> 374 us).
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

// Biased exponent of a row's largest value; the range in which every scaled
// quantity of a product stays a normal FP64 number.  Rows outside it (and rows
// with values that are not finite) are multiplied in FP64: kX64Native, an
// exponent so large that their digits are zeros.
constexpr int kExpLo = 1023 - 800, kExpHi = 1023 + 800, kExpOff = 1080, kX64Native = 4000;
__device__ __forceinline__ int exponent_of(unsigned key) {   // of the row's largest key, see Tile
    const int e = (int)(key >> 5);
    return key == 0 ? kExpLo : (e >= kExpLo && e <= kExpHi ? e : kX64Native);
}

// v = round(x * 2^(1080 - eref)), |v| < 2^58 where x's exponent is at most eref
// (and eref at least kExpLo: a subnormal's missing leading bit is far below the
// unit), as 2 (v + bias), or 1 more.
constexpr u64 kBias = 512 * (1ull + (1ull << 10) + (1ull << 20) + (1ull << 30) + (1ull << 40) + (1ull << 50));
__device__ __forceinline__ u64 to_fixed(double x, int eref) {
    const int hi = __double2hiint(x), neg = hi >> 31;
    const unsigned lo = (unsigned)__double2loint(x);
    const u64 m = ((u64)(((unsigned)hi & 0xfffffu) | 0x100000u) << 32 | lo) << 6;
    const int d = min(eref - ((hi >> 20) & 0x7ff), 63);
    return ((m >> d) ^ (u64)(i64)neg) + (2 * kBias + 1 - (u64)(i64)neg);
}
// 2 (v 2^sh + bias) for an integer, rounded likewise (|v| 2^sh <= 2^58).
__device__ __forceinline__ u64 shifted(i64 v, int sh) {
    const int l = min(max(sh + 1, 0), 31), r = min(max(-(sh + 1), 0), 63);
    return (u64)((v << l) >> r) + (2 * kBias + 1);
}
// v * 2^e, correctly rounded (the result is a normal number).
__device__ __forceinline__ double to_double(i64 v, int e) {
    const double x = (double)v;
    const int hi = __double2hiint(x);
    return __hiloint2double(hi ? hi + (e << 20) : 0, __double2loint(x));   // hi = 0: v = 0
}
// The same in integer instructions, about 25 (|v| < 2^61).
__device__ __forceinline__ double to_double_int(i64 v, int e) {
    const u64 a = (u64)(v < 0 ? -v : v);
    const int z = __clzll((i64)a) - 1;   // the leading bit goes to 62
    const u64 r = (((a << z) + 512) >> 10) + ((u64)(unsigned)(e + 1084 - z) << 52);   // 2^52 <= first part <= 2^53
    const unsigned hi = (unsigned)(r >> 32) | ((unsigned)(v >> 32) & 0x80000000u);
    return a == 0 ? 0.0 : __hiloint2double((int)hi, (int)(unsigned)r);
}
__device__ __forceinline__ i64 shr_round(i64 v, int s) {   // v / 2^s, s >= 0
    s = s > 62 ? 62 : s;
    return (v + ((1LL << s) >> 1)) >> s;
}

// Digits of a pair of such values at k = 2t, 2t + 1, as half2 words: the unsigned
// digits of v + bias, in [0, 2^60), are 512 above the balanced ones.
__device__ __forceinline__ void digits(u64 a, u64 b, unsigned (&d)[kX64Digits]) {
    const unsigned al = (unsigned)a, ah = (unsigned)(a >> 32), bl = (unsigned)b, bh = (unsigned)(b >> 32);
    const unsigned x[kX64Digits] = {ah >> 19, ah >> 9, __funnelshift_r(al, ah, 31), al >> 21, al >> 11, al >> 1};
    const unsigned y[kX64Digits] = {bh >> 19, bh >> 9, __funnelshift_r(bl, bh, 31), bl >> 21, bl >> 11, bl >> 1};
#pragma unroll
    for (int i = 0; i < kX64Digits; ++i) {
        const unsigned w = (__byte_perm(x[i], y[i], 0x5410) & 0x03ff03ffu) | 0x64006400u;   // 1024 + digit
        asm("add.f16x2 %0, %1, %2;" : "=r"(d[i]) : "r"(w), "r"(0xe600e600u));               // - 1536
    }
}

// The digits of a tile: rows g (h = 0) and g + 8 (h = 1), one or two groups of 8
// operands, each lane holding 2t and 2t + 1 of every group; e[h]: the row's
// exponent.
template <int K>
struct Tile {
    static constexpr int KG = (K + 7) / 8;
    unsigned a[KG][kX64Digits][2];
    int e[2];
    // ld0(k), ld1(k): operand k of this lane's row 0, 1 (0 outside the row)
    template <typename LD0, typename LD1>
    __device__ __forceinline__ void fill(int t, LD0 ld0, LD1 ld1) {
        double v[2][2 * KG];
        unsigned m = 0, z0 = 0, z1 = 0;   // m: exponents and leading mantissa bits, 16 bits a row
#pragma unroll
        for (int k = 0; k < 2 * KG; ++k) {
            const int kk = 8 * (k >> 1) + 2 * t + (k & 1);
            v[0][k] = ld0(kk);
            v[1][k] = ld1(kk);
            const unsigned h0 = (unsigned)__double2hiint(v[0][k]) << 1, h1 = (unsigned)__double2hiint(v[1][k]) << 1;
            m = __vmaxu2(m, __byte_perm(h0, h1, 0x7632));
            z0 |= h0 | (unsigned)__double2loint(v[0][k]);
            z1 |= h1 | (unsigned)__double2loint(v[1][k]);
        }
        m |= min(z0, 1u) | min(z1, 1u) << 16;   // 0 for a row of zeros only
        m = __vmaxu2(m, __shfl_xor_sync(0xffffffffu, m, 1));   // over the four lanes that hold the rows
        m = __vmaxu2(m, __shfl_xor_sync(0xffffffffu, m, 2));
        e[0] = exponent_of(m & 0xffffu);
        e[1] = exponent_of(m >> 16);
        split([&](int h, int k) { return to_fixed(v[h][k], e[h]); });
    }
    // The same from integers: operand k of row h is v 2^x, v = ld0(k), ld1(k), x = x0[j], x1[j] for this
    // lane's j-th operand.
    template <typename LD0, typename LD1>
    __device__ __forceinline__ void fill_int(int t, LD0 ld0, LD1 ld1, const int (&x0)[2 * KG], const int (&x1)[2 * KG]) {
        i64 v[2][2 * KG];
        unsigned m = 0x80008000u;   // exponents of the operands' leading bits, 16 bits a row
#pragma unroll
        for (int k = 0; k < 2 * KG; ++k) {
            const int kk = 8 * (k >> 1) + 2 * t + (k & 1);
            v[0][k] = ld0(kk);
            v[1][k] = ld1(kk);
            const int q0 = v[0][k] == 0 ? -30000 : x0[k] - __clz(abs_hi(v[0][k])),
                      q1 = v[1][k] == 0 ? -30000 : x1[k] - __clz(abs_hi(v[1][k]));
            m = __vmaxs2(m, __byte_perm((unsigned)q0, (unsigned)q1, 0x5410));
        }
        m = __vmaxs2(m, __shfl_xor_sync(0xffffffffu, m, 1));
        m = __vmaxs2(m, __shfl_xor_sync(0xffffffffu, m, 2));
        const int q[2] = {(int)(short)(m & 0xffffu), (int)m >> 16};
        e[0] = q[0] + kExpOff + 6;
        e[1] = q[1] + kExpOff + 6;
        split([&](int h, int k) { return shifted(v[h][k], (h ? x1[k] : x0[k]) - q[h] - 6); });
    }
    __device__ __forceinline__ bool native() const { return e[0] == kX64Native || e[1] == kX64Native; }
    // exponent of the products of row h with an operator of scale s, and a product's value
    __device__ __forceinline__ int exponent(int h, int s) const { return e[h] - kExpOff + s; }
    __device__ __forceinline__ double value(i64 o, int h, int s) const { return to_double(o, exponent(h, s)); }

  private:
    template <typename F>
    __device__ __forceinline__ void split(F f) {
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int g = 0; g < KG; ++g) {
                unsigned d[kX64Digits];
                digits(f(h, 2 * g), f(h, 2 * g + 1), d);
#pragma unroll
                for (int i = 0; i < kX64Digits; ++i) a[g][i][h] = d[i];
            }
    }
    // magnitude bits of the high word
    static __device__ __forceinline__ int abs_hi(i64 v) { return (int)(v >> 32) ^ (int)(v >> 63); }
};
struct ZeroRow {   // (its digits are known when the kernel is compiled)
    __device__ __forceinline__ i64 operator()(int) const { return 0; }
};
// Exponents of a lane's operands, each of a row of its own in the tiles they were written from: w[g]
// the exponent of row g, 16 bits (HI: the upper ones), held by that row's lanes.
template <int KG, bool HI>
__device__ __forceinline__ void operand_exponents(const unsigned (&w)[KG], int t, int (&x)[2 * KG]) {
#pragma unroll
    for (int k = 0; k < 2 * KG; ++k) {
        const unsigned u = __shfl_sync(0xffffffffu, w[k >> 1], 4 * (2 * t + (k & 1)));
        x[k] = HI ? (int)u >> 16 : (int)(short)(u & 0xffffu);
    }
}
__device__ __forceinline__ unsigned pack16(int lo, int hi) { return __byte_perm((unsigned)lo, (unsigned)hi, 0x5410); }

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
// o[2 h + c] = the value of row (h) and column 8 nt + 2 t + c.
template <int K>
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
}

// sum_m R[m rs] v[m vs], for the rows that the digits cannot hold (not inlined:
// it must not cost the kernels registers).
static __device__ __noinline__ double x64_native_row(const double* v, int vs, const double* R, int rs, int n) {
    double s = 0.0;
    for (int m = 0; m < n; ++m) s += R[m * rs] * v[m * vs];
    return s;
}

// One volume pass over the N^2 pencils along direction dir: out (or, acc, out +=)
// R in, R with digit words op and scale s; M, mr, mc: R in FP64 (R[i][m] = M[i mr + m mc]).
// The tiles of 16 pencils are dealt to the CTA's warps, from warp w on.  One
// function for all twelve passes: inlined, they outgrow the instruction cache
// (7,680 hp elements, n = 8: element kernel 177 against 145 us).
template <int N, int W>
__device__ __noinline__ void x64_pass(const double* __restrict__ in, double* __restrict__ out, int dir,
                                      const unsigned* __restrict__ op, int s, const double* __restrict__ M, int mr,
                                      int mc, bool acc, int w) {
    constexpr int NN = N * N, TILES = (NN + 15) / 16, NT = (N + 7) / 8;
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const int stride = dir == 0 ? 1 : (dir == 1 ? Strides<N>::S1 : Strides<N>::S2);
    const int su = dir == 0 ? Strides<N>::S1 : 1, sv = dir == 2 ? Strides<N>::S1 : Strides<N>::S2;
    unsigned native = 0;
#pragma unroll 1   // (two tiles at a time: no faster)
    for (int j = 0; j < (TILES + W - 1) / W; ++j) {
        const int tile = w + j * W;
        if (TILES % W != 0 && tile >= TILES) continue;
        const int p0 = 16 * tile + g, p1 = p0 + 8;
        const bool v0 = p0 < NN, v1 = p1 < NN;
        const int b0 = v0 ? su * (p0 % N) + sv * (p0 / N) : 0, b1 = v1 ? su * (p1 % N) + sv * (p1 / N) : 0;
        Tile<N> A;
        A.fill(t, [&](int k) { return v0 && k < N ? in[b0 + k * stride] : 0.0; },
               [&](int k) { return v1 && k < N ? in[b1 + k * stride] : 0.0; });
        native |= ((A.e[0] == kX64Native ? 1u : 0u) | (A.e[1] == kX64Native ? 2u : 0u)) << (2 * j);
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
            i64 o[4];
            tile_product<N>(A, op, nt, lane, o);
#pragma unroll
            for (int h = 0; h < 2; ++h)
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    const int col = 8 * nt + 2 * t + c;
                    if (!(h ? v1 : v0) || col >= N) continue;
                    const int idx = (h ? b1 : b0) + col * stride;
                    const double v = N > 8 ? A.value(o[2 * h + c], h, s) : to_double_int(o[2 * h + c], A.exponent(h, s));
                    out[idx] = acc ? out[idx] + v : v;
                }
        }
    }
    if (native)   // rows in FP64 (their digits were zero: nothing, or 0, is in their place)
        for (int j = 0; j < 2 * ((TILES + W - 1) / W); ++j)
            if (native >> j & 1) {
                const int p = 16 * (w + (j >> 1) * W) + 8 * (j & 1) + g, b = su * (p % N) + sv * (p / N);
                for (int nt = 0; nt < NT; ++nt)
                    for (int col = 8 * nt + 2 * t; col < min(N, 8 * nt + 2 * t + 2); ++col)
                        out[b + col * stride] += x64_native_row(in + b, stride, M + col * mr, mc, N);
            }
}

// Trace of one mortar side in FP64 from the element's values U and its normal
// derivatives D on the face (see x64_trace_slot).
static __device__ __noinline__ void x64_native_trace(const double* U, const double* D, int st1, int st2, int n, int q,
                                                     int o, const double* M1, const double* M2, const double* c1,
                                                     const double* c2, const double* cn, double* out, double* X,
                                                     int lane) {
    const int q2 = q * q;
    double *U1 = X, *D1 = U1 + q * n, *N1 = D1 + q * n;
    for (int k = lane; k < q * n; k += 32) {
        const int i1 = k % q, b = k / q;
        double su = 0, sd = 0, sn = 0;
        for (int a = 0; a < n; ++a) {
            const double iv = M1[2 * (i1 * n + a)], dv = M1[2 * (i1 * n + a) + 1], u = U[a * st1 + b * st2];
            su += iv * u;
            sd += dv * u;
            sn += iv * D[a + n * b];
        }
        U1[k] = su;
        D1[k] = sd;
        N1[k] = sn;
    }
    __syncwarp();
    for (int k = lane; k < q2; k += 32) {
        const int i1 = k % q, i2 = k / q;
        const int b1 = (o & 2) ? q - 1 - i1 : i1, b2 = (o & 4) ? q - 1 - i2 : i2;
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
        out[q2 + kA] = c1[kA] * g1 + c2[kA] * g2 + cn[kA] * gn;
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

// ---- trace kernel -------------------------------------------------------------------
// Shared memory of an element's CTA (in 8-byte values).
template <int N, int W>
struct X64Layout {
    static constexpr int NR = r4(Strides<N>::SIZE), OPW = x64_op_words(N, N) / 2;
    static constexpr int TTAB = OPW + r4(N * N);                    // DL ends' digits, DL
    static constexpr int TDF = 6 * N * N, TSCR = 3 * kQ * N;        // normal derivatives on the faces; per warp
    static constexpr int TSIZE = r4(TTAB + NR + TDF + W * TSCR);
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

// Trace of this side at the Q x Q mortar points from the element's values U and
// its normal derivatives D on the face (see trace_slot).
template <int N, int QM>
__device__ __forceinline__ void x64_trace_slot(const SlotInfo<double>& s, const double* __restrict__ U,
                                               const double* __restrict__ D, const unsigned* __restrict__ FW,
                                               const int* __restrict__ FS, const double* __restrict__ ftab, double* X,
                                               const double* __restrict__ co, double* __restrict__ mt, int lane) {
    constexpr int NTQ = (QM + 7) / 8, HN = (N + 7) / 8, HQ = (QM + 7) / 8;
    const int Q = s.q, Q2 = Q * Q;
    const int d = s.f >> 1, fn = (s.f & 1) ? N - 1 : 0, g = lane >> 2, t = lane & 3;
    int t1, t2;
    tangential(d, t1, t2);
    const int st1 = stride_of<N>(t1), st2 = stride_of<N>(t2);
    U += fn * stride_of<N>(d);
    D += fn ? N * N : 0;
    double* out = mt + 4 * s.goff + 2 * s.side * Q2;
    const unsigned* I1 = x64_face_op<N, QM>(FW, Q, s.p0, 0);
    const unsigned* D1 = x64_face_op<N, QM>(FW, Q, s.p0, 1);
    const unsigned* I2 = x64_face_op<N, QM>(FW, Q, s.p1, 0);
    const unsigned* D2 = x64_face_op<N, QM>(FW, Q, s.p1, 1);
    const int sI = FS[x64_face_scale(N, Q)], sD = FS[x64_face_scale(N, Q) + 1];
    i64 *XU = reinterpret_cast<i64*>(X), *XD = XU + Q * N, *XN = XD + Q * N;   // [i1 + Q b]
    unsigned xe[HN];   // exponents of row b's products with I: of U, of D
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
    bool native = false;
#pragma unroll
    for (int hb = 0; hb < HN; ++hb) {
        const int b = 8 * hb + g;
        const bool v = b < N;
        Tile<N> A;
        A.fill(t, [&](int k) { return v && k < N ? U[k * st1 + b * st2] : 0.0; },
               [&](int k) { return v && k < N ? D[k + N * b] : 0.0; });
        native |= A.native();
        xe[hb] = pack16(A.exponent(0, sI), A.exponent(1, sI));
#pragma unroll
        for (int nt = 0; nt < NTQ; ++nt) {
            i64 o[4], e[4];
            tile_product<N>(A, I1, nt, lane, o);
            tile_product<N>(A, D1, nt, lane, e);
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                const int i1 = 8 * nt + 2 * t + c;
                if (v && i1 < Q) {
                    XU[i1 + Q * b] = o[c];
                    XN[i1 + Q * b] = o[2 + c];
                    XD[i1 + Q * b] = e[c];
                }
            }
        }
    }
    __syncwarp();
    int xu[2 * HN], xd[2 * HN], xn[2 * HN];
    operand_exponents<HN, false>(xe, t, xu);
    operand_exponents<HN, true>(xe, t, xn);
#pragma unroll
    for (int k = 0; k < 2 * HN; ++k) xd[k] = xu[k] + sD - sI;
#pragma unroll
    for (int hq = 0; hq < HQ; ++hq) {
        const int i1 = 8 * hq + g;
        const bool v = i1 < Q;
        Tile<N> A, B;
        A.fill_int(t, [&](int k) { return v && k < N ? XU[i1 + Q * k] : 0LL; },
                   [&](int k) { return v && k < N ? XD[i1 + Q * k] : 0LL; }, xu, xd);
        B.fill_int(t, [&](int k) { return v && k < N ? XN[i1 + Q * k] : 0LL; }, ZeroRow(), xn, xn);
#pragma unroll
        for (int nt = 0; nt < NTQ; ++nt) {
            i64 o[4], e[4], w[4];
            tile_product<N>(A, I2, nt, lane, o);
            tile_product<N>(A, D2, nt, lane, e);
            tile_product<N>(B, I2, nt, lane, w);
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                const int i2 = 8 * nt + 2 * t + c;
                if (v && i2 < Q) {
                    const int kA = x64_point(s.o, Q, i1, i2);
                    out[kA] = A.value(o[c], 0, sI);
                    const double c1 = QM == 8 ? cv[c][0] : co[t1 * Q2 + kA], c2 = QM == 8 ? cv[c][1] : co[t2 * Q2 + kA],
                                 cn = QM == 8 ? cv[c][2] : co[d * Q2 + kA];
                    out[Q2 + kA] = c1 * A.value(o[2 + c], 1, sI) + c2 * A.value(e[c], 0, sD) + cn * B.value(w[c], 0, sI);
                }
            }
        }
    }
    __syncwarp();
    if (__any_sync(0xffffffffu, native))   // (in the place of what was written above)
        x64_native_trace(U, D, st1, st2, N, Q, s.o, ftab + face_tab_off(N, Q, s.p0), ftab + face_tab_off(N, Q, s.p1),
                         co + t1 * Q2, co + t2 * Q2, co + d * Q2, out, X, lane);
}

// One CTA per element, elements blk, blk + nblk, ... of the bucket.
template <int N, int W>
__device__ __forceinline__ void x64_trace_body(const LevelView<double>& L, const ElemDesc* __restrict__ bdesc,
                                               int count, const double* __restrict__ x, int blk, int nblk) {
    using Ly = X64Layout<N, W>;
    constexpr int N3 = N * N * N, R = (N3 + (32 * W) - 1) / (32 * W), TILES = (N * N + 15) / 16;
    extern __shared__ __align__(16) double x64_smem[];
    unsigned* sW = reinterpret_cast<unsigned*>(x64_smem);
    double* sDL = x64_smem + Ly::OPW;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
    for (int k = tid; k < x64_op_words(2, N); k += (32 * W)) sW[k] = L.x64.w[x64_vol_off(N, kX64Ends) + k];
    for (int k = tid; k < N * N; k += (32 * W)) sDL[k] = L.tab[tab_n(TabIndex::DL, N) + k];
    const int sE = L.x64.s[x64_vol_scale(N) + kX64Ends];
    double* U = x64_smem + Ly::TTAB;
    double* DF = U + Ly::NR;                     // [direction][face][N^2]
    double* X = DF + Ly::TDF + warp * Ly::TSCR;
    for (int ei = blk; ei < count; ei += nblk) {
        const ElemDesc de = bdesc[ei];
        WarpSlots<double> ws;
        ws.load(L, de.s0, de.s1, lane);
        double v[R];
#pragma unroll
        for (int j = 0; j < R; ++j) v[j] = tid + (32 * W) * j < N3 ? x[de.dofo + tid + (32 * W) * j] : 0.0;
        if (warp == 0) ws.prefetch(L, lane, false);
        __syncthreads();   // the previous element's slots are done
#pragma unroll
        for (int j = 0; j < R; ++j) {
            const int k = tid + (32 * W) * j;
            if (k < N3) U[sidx<N>(k)] = v[j];
        }
        __syncthreads();
        // face-normal derivatives of the six faces: the tiles of the three directions dealt to the warps
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
                A.fill(t, [&](int k) { return v0 && k < N ? U[b0 + k * sd] : 0.0; },
                       [&](int k) { return v1 && k < N ? U[b1 + k * sd] : 0.0; });
                i64 o[4];
                tile_product<N>(A, sW, 0, lane, o);
                if (t == 0) {   // columns 0, 1: the two faces
                    double* D = DF + 2 * d * N * N;
#pragma unroll
                    for (int h = 0; h < 2; ++h)
#pragma unroll
                        for (int c = 0; c < 2; ++c)
                            if (h ? v1 : v0)
                                D[c * N * N + (h ? p1 : p0)] =
                                    A.e[h] == kX64Native ? x64_native_row(U + (h ? b1 : b0), sd, sDL + c * (N - 1) * N, 1, N)
                                                         : A.value(o[2 * h + c], h, sE);
                }
            }
        }
        __syncthreads();
        const double* ft = L.ftab + face_seg_off(N);
        for (int si = ws.s0 + warp; si < ws.s1; si += W) {
            const SlotInfo<double> s = unpack_rec(ws.get(si));
            const double* D = DF + 2 * (s.f >> 1) * N * N;
            const double* co = L.mg + 7 * s.goff + (s.side == 0 ? 1 : 4) * s.q * s.q;
            if (N <= 8 && s.q <= 8)
                x64_trace_slot<N, (N > 8 ? 9 : 8)>(s, U, D, L.x64.w, L.x64.s, ft, X, co, L.mt, lane);
            else
                x64_trace_slot<N, 9>(s, U, D, L.x64.w, L.x64.s, ft, X, co, L.mt, lane);
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
    // QM = 8: a lane needs the fluxes of two points only, (g, 2t) and (g, 2t + 1), and keeps them in registers
    double pv[2][4] = {{0, 0, 0, 0}, {0, 0, 0, 0}};
    if constexpr (QM == 8) {
#pragma unroll
        for (int c = 0; c < 2; ++c)
            if (g < Q && 2 * t + c < Q) flux(g, 2 * t + c, pv[c]);
    } else {
        for (int k = lane; k < Q2; k += 32) {
            double p[4];
            flux(k % Q, k / Q, p);
            PA[k] = p[0];
            P1[k] = p[1];
            P2[k] = p[2];
            Pn[k] = p[3];
        }
        __syncwarp();
    }
    const unsigned* I1 = x64_face_op<N, QM>(FW, Q, s.p0, 2);
    const unsigned* D1 = x64_face_op<N, QM>(FW, Q, s.p0, 3);
    const unsigned* I2 = x64_face_op<N, QM>(FW, Q, s.p1, 2);
    const unsigned* D2 = x64_face_op<N, QM>(FW, Q, s.p1, 3);
    const int sI = FS[x64_face_scale(N, Q) + 2], sD = FS[x64_face_scale(N, Q) + 3];
    double* Xd = F + 4 * Q2;
    i64 *X1 = reinterpret_cast<i64*>(Xd), *X2 = X1 + Q * N, *X3 = X2 + Q * N;   // [i1 + Q b]
    unsigned xe[HQ], x3e[HQ];   // exponents of row i1: of X1 and X2, of X3
    bool native = false;
#pragma unroll
    for (int hq = 0; hq < HQ; ++hq) {
        const int i1 = 8 * hq + g;
        const bool v = i1 < Q;
        Tile<QM> A, B;
        auto at = [&](const double* P, int i, int k) { return QM == 8 ? pv[k & 1][i] : (v && k < Q ? P[i1 + Q * k] : 0.0); };
        A.fill(t, [&](int k) { return at(PA, 0, k); },
               [&](int k) { return at(P1, 1, k); });
        B.fill(t, [&](int k) { return at(Pn, 3, k); },
               [&](int k) { return at(P2, 2, k); });
        native |= A.native() || B.native();
        const int exA = A.exponent(0, sI), exD = B.exponent(1, sD), ex1 = max(exA, exD) + 1;   // X1 = I^T PA + D^T P2
        xe[hq] = pack16(ex1, A.exponent(1, sI));
        x3e[hq] = (unsigned)B.exponent(0, sI);
#pragma unroll
        for (int nt = 0; nt < NTN; ++nt) {
            i64 o[4], w[4], e[4];
            tile_product<QM>(A, I2, nt, lane, o);
            tile_product<QM>(B, I2, nt, lane, w);
            tile_product<QM>(B, D2, nt, lane, e);
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                const int b = 8 * nt + 2 * t + c;
                if (v && b < N) {
                    X1[i1 + Q * b] = shr_round(o[c], ex1 - exA) + shr_round(e[2 + c], ex1 - exD);
                    X2[i1 + Q * b] = o[2 + c];
                    X3[i1 + Q * b] = w[c];
                }
            }
        }
    }
    __syncwarp();
    int x1[2 * HQ], x2[2 * HQ], x3[2 * HQ];
    operand_exponents<HQ, false>(xe, t, x1);
    operand_exponents<HQ, true>(xe, t, x2);
    operand_exponents<HQ, false>(x3e, t, x3);
    if (__any_sync(0xffffffffu, native)) {
        const double* ft = L.ftab + face_seg_off(N);
        __syncwarp();
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
#pragma unroll
    for (int hb = 0; hb < HN; ++hb) {
        const int b = 8 * hb + g;
        const bool v = b < N;
        Tile<QM> A, B;
        A.fill_int(t, [&](int k) { return v && k < Q ? X1[k + Q * b] : 0LL; },
                   [&](int k) { return v && k < Q ? X3[k + Q * b] : 0LL; }, x1, x3);
        B.fill_int(t, [&](int k) { return v && k < Q ? X2[k + Q * b] : 0LL; }, ZeroRow(), x2, x2);
#pragma unroll
        for (int nt = 0; nt < NTN; ++nt) {
            i64 o[4], w[4];
            tile_product<QM>(A, I1, nt, lane, o);
            tile_product<QM>(B, D1, nt, lane, w);
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                const int a = 8 * nt + 2 * t + c;
                if (v && a < N) {
                    const double fu = A.value(o[c], 0, sI) + B.value(w[c], 0, sD), fd = A.value(o[2 + c], 1, sI);
                    FU[a + N * b] = first ? fu : FU[a + N * b] + fu;
                    FD[a + N * b] = first ? fd : FD[a + N * b] + fd;
                }
            }
        }
    }
    __syncwarp();
}

// Volume terms of one element into Y, by the whole CTA (I and Dg: the operators
// in FP64, for rows that the digits cannot hold).  Ends with a barrier.
template <int N, int W>
__device__ __forceinline__ void x64_volume(const double* __restrict__ x, const double* __restrict__ Ge,
                                           const double* __restrict__ c0e, const unsigned* sW, int sI, int sIT, int sD,
                                           int sDT, const double* __restrict__ I, const double* __restrict__ Dg,
                                           double* Y, double* A, double* G1, double* U) {
    constexpr int N3 = N * N * N, R = (N3 + (32 * W) - 1) / (32 * W), OPW = x64_op_words(N, N),
                  TILES = (N * N + 15) / 16;
    const int tid = threadIdx.x, warp = tid >> 5;
    const unsigned *wI = sW, *wIT = wI + OPW, *wD = wIT + OPW, *wDT = wD + OPW;
    {
        double v[R];
#pragma unroll
        for (int j = 0; j < R; ++j) v[j] = tid + (32 * W) * j < N3 ? x[tid + (32 * W) * j] : 0.0;
        prefetch_l2(Ge, 6 * N3, tid, (32 * W));   // metric terms, needed after 6 passes
#pragma unroll
        for (int j = 0; j < R; ++j) {
            const int k = tid + (32 * W) * j;
            if (k < N3) U[sidx<N>(k)] = v[j];
        }
    }
    __syncthreads();
    x64_pass<N, W>(U, A, 0, wI, sI, I, N, 1, false, warp);
    __syncthreads();
    x64_pass<N, W>(A, G1, 1, wI, sI, I, N, 1, false, warp);
    __syncthreads();
    x64_pass<N, W>(G1, A, 2, wI, sI, I, N, 1, false, warp);
    __syncthreads();
    x64_pass<N, W>(A, G1, 0, wD, sD, Dg, N, 1, false, warp);
    x64_pass<N, W>(A, Y, 1, wD, sD, Dg, N, 1, false, (warp + TILES) % W);
    x64_pass<N, W>(A, U, 2, wD, sD, Dg, N, 1, false, (warp + 2 * TILES) % W);
    __syncthreads();
    for (int k = tid; k < N3; k += (32 * W)) {
        const int s = sidx<N>(k);
        const double m00 = __ldcs(Ge + k), m01 = __ldcs(Ge + N3 + k), m02 = __ldcs(Ge + 2 * N3 + k);
        const double m11 = __ldcs(Ge + 3 * N3 + k), m12 = __ldcs(Ge + 4 * N3 + k), m22 = __ldcs(Ge + 5 * N3 + k);
        const double g0 = G1[s], g1 = Y[s], g2 = U[s];
        G1[s] = m00 * g0 + m01 * g1 + m02 * g2;
        Y[s] = m01 * g0 + m11 * g1 + m12 * g2;
        U[s] = m02 * g0 + m12 * g1 + m22 * g2;
        if (c0e) A[s] = c0e[k] * A[s];
    }
    __syncthreads();
    x64_pass<N, W>(G1, A, 0, wDT, sDT, Dg, 1, N, c0e != nullptr, warp);
    __syncthreads();
    x64_pass<N, W>(Y, A, 1, wDT, sDT, Dg, 1, N, true, warp);
    __syncthreads();
    x64_pass<N, W>(U, A, 2, wDT, sDT, Dg, 1, N, true, warp);
    __syncthreads();
    x64_pass<N, W>(A, G1, 0, wIT, sIT, I, 1, N, false, warp);
    __syncthreads();
    x64_pass<N, W>(G1, U, 1, wIT, sIT, I, 1, N, false, warp);
    __syncthreads();
    x64_pass<N, W>(U, Y, 2, wIT, sIT, I, 1, N, false, warp);
    __syncthreads();
}

// Degrees whose volume terms stay in FP64: a pass of the integers takes the
// time of a tile (about 1.5 us of latency) however few pencils it has, and
// 12 n^4 FP64 multiply-adds are fewer than that up to n = 5 (4,096 elements of p =
// 4: 230 us, 246 on digits; 512: 50 and 56).
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
        if constexpr (x64_small<N>())
            x64_small_volume<N, W>(x + de.dofo, Ge, c0e, x64_smem, x64_smem + N2, Y, A, G1, U);
        else
            x64_volume<N, W>(x + de.dofo, Ge, c0e, sW, sI, sIT, sD, sDT, L.tab + tab_n(TabIndex::I, N),
                             L.tab + tab_n(TabIndex::Dg, N), Y, A, G1, U);
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
