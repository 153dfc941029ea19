// 64-bit fixed-point evaluation of the 3D nonlinear-diffusion (residual and
// vector-Jacobian product), 2D Bratu and 2D minimal-surface elements, for the FP64 kernels.
//
// What bounds an FP64 element kernel on this GPU is the FP64 pipe: 2
// operations per clock and SM.  The integer pipe adds 64-bit integers at ~52
// and multiplies 32 x 32 -> 64 bit at ~24 per clock and SM (measured), so the
// element arithmetic of element.cuh runs here on 64-bit integers under a block
// exponent per element, and only the conversions' exponents and the sums over
// elements are FP64.
//
// Precision.  The corner values of an element are shifted to the exponent of
// the largest, with two bits below its last place: exact for every corner
// within a factor 4 of the largest, and otherwise off by less than 2^-55 of
// it (the differences, which are what is computed with, are then of the
// largest's size).  All butterflies are exact.  The modes that carry the
// gradient are left-aligned once more, exactly, so that the largest has 61
// bits whatever the smoothness of the field; products keep the upper 64 of 128
// bits.
//
// The FP64 pipe also runs the hardware conversions between FP64 and 64-bit
// integers (17 conversions an element took as long as the arithmetic), so the
// values enter by shifts: a node value is packed once as significand and
// exponent, and an element shifts its 8 corners to their common exponent.
#pragma once
#include <stdint.h>
#include <string.h>

#include "fx_tables.cuh"

#ifndef __CUDACC__
#include <cmath>
#ifndef __host__
#define __host__
#define __device__
#define __forceinline__ inline
#endif
#endif

namespace jfnk {

typedef long long fx_t;

#ifdef __CUDACC__
static __device__ const fx_t kFxExp2Dev[256] = {JFNK_FX_EXP2_TABLE};
#endif
static const fx_t kFxExp2Host[256] = {JFNK_FX_EXP2_TABLE};

__host__ __device__ __forceinline__ int fx_hi(fx_t a) { return (int)(a >> 32); }
__host__ __device__ __forceinline__ unsigned int fx_lo(fx_t a) { return (unsigned int)a; }

__host__ __device__ __forceinline__ int fx_mulhi_s(int a, int b) {
#ifdef __CUDA_ARCH__
    return __mulhi(a, b);
#else
    return (int)(((long long)a * b) >> 32);
#endif
}
// upper word of a b, plus c
__host__ __device__ __forceinline__ int fx_madhi_s(int a, int b, int c) {
#ifdef __CUDA_ARCH__
    int d;
    asm("mad.hi.s32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
    return d;
#else
    return fx_mulhi_s(a, b) + c;
#endif
}
// arithmetic shift right, by 63 at most
__host__ __device__ __forceinline__ fx_t fx_sar(fx_t a, int s) {
#ifdef __CUDA_ARCH__
    fx_t d;
    asm("shr.s64 %0, %1, %2;" : "=l"(d) : "l"(a), "r"(s));  // clamps the shift
    return d;
#else
    return a >> (s > 63 ? 63 : s);
#endif
}
__host__ __device__ __forceinline__ unsigned int fx_mulhi_u(unsigned int a, unsigned int b) {
#ifdef __CUDA_ARCH__
    return __umulhi(a, b);
#else
    return (unsigned int)(((unsigned long long)a * b) >> 32);
#endif
}
__host__ __device__ __forceinline__ int fx_clz(unsigned int a) {
#ifdef __CUDA_ARCH__
    return __clz((int)a);
#else
    return a ? __builtin_clz(a) : 32;
#endif
}
__host__ __device__ __forceinline__ fx_t fx_shl(fx_t a, int s) { return (fx_t)((unsigned long long)a << s); }
// round to nearest integer of a double below 2^62 in magnitude
__host__ __device__ __forceinline__ fx_t fx_rint(double a) {
#ifdef __CUDA_ARCH__
    return __double2ll_rn(a);
#else
    return (fx_t)std::llrint(a);
#endif
}
__host__ __device__ __forceinline__ double fx_double(fx_t a) {
#ifdef __CUDA_ARCH__
    return __ll2double_rn(a);
#else
    return (double)a;
#endif
}
__host__ __device__ __forceinline__ long long dbl_bits(double a) {
#ifdef __CUDA_ARCH__
    return __double_as_longlong(a);
#else
    long long b;
    memcpy(&b, &a, 8);
    return b;
#endif
}
__host__ __device__ __forceinline__ int dbl_hi(double a) {
#ifdef __CUDA_ARCH__
    return __double2hiint(a);
#else
    long long b;
    memcpy(&b, &a, 8);
    return (int)(b >> 32);
#endif
}
__host__ __device__ __forceinline__ double dbl_addexp(double a, int hi_add) {
#ifdef __CUDA_ARCH__
    return __hiloint2double(__double2hiint(a) + hi_add, __double2loint(a));
#else
    long long b;
    memcpy(&b, &a, 8);
    b += (long long)((unsigned long long)(unsigned int)hi_add << 32);
    memcpy(&a, &b, 8);
    return a;
#endif
}

// A positive multiplier below 2^63 as h 2^32 + l with a signed lower half.
struct FxMul {
    int h, l;
};
__host__ __device__ __forceinline__ FxMul fx_split(fx_t b) {
    const fx_t c = b + (fx_t)0x80000000LL;
    return {fx_hi(c), (int)(fx_lo(c) ^ 0x80000000u)};
}
// a b / 2^64, less than 3 off: the product of the lower halves is left out and
// the cross terms are truncated.  The two cross terms' sum has to fit a signed
// word: |a| / 2^33 + b / 2^32 < 2^31.
__host__ __device__ __forceinline__ fx_t fx_mul(fx_t a, FxMul b) {
    const int t = fx_madhi_s(fx_hi(a), b.l, (int)fx_mulhi_u(fx_lo(a), (unsigned int)b.h));
    return (fx_t)fx_hi(a) * b.h + t;
}

// a b / 2^64 of two split numbers, less than 2 off
__host__ __device__ __forceinline__ fx_t fx_mul(FxMul a, FxMul b) {
    return (fx_t)a.h * b.h + fx_madhi_s(a.h, b.l, fx_mulhi_s(a.l, b.h));
}

// 1/sqrt 3, 1/3 and 1/(3 sqrt 3), times 2^63
constexpr fx_t kFxA1 = 0x49e69d1640cc7135LL, kFxA2 = 0x2aaaaaaaaaaaaaabLL, kFxA3 = 0x18a2345cc04425bcLL;

// Test-side multipliers of an element: A^k times a positive scale (the node
// factor, and kappa), its power of two apart.  b_k = A^k m 2^63 (b0: m 2^62),
// scale = m 2^ex with m in [1/2, 1).
struct FxScale {
    FxMul b0, b1, b2, b3;
    int ex;
};
// a positive normal double as m 2^62 (exact) and ex
__host__ __device__ __forceinline__ FxMul fx_significand(double x, int& ex) {
    ex = (dbl_hi(x) >> 20) - 1022;
    return fx_split(fx_rint(dbl_addexp(x, (62 - ex) * (1 << 20))));
}
__host__ __device__ __forceinline__ FxScale fx_scale(double scale) {
    FxScale s;
    const FxMul m = fx_significand(scale, s.ex);
    s.b0 = m;
    s.b1 = fx_split(fx_shl(fx_mul(kFxA1, m), 2));
    s.b2 = fx_split(fx_shl(fx_mul(kFxA2, m), 2));
    s.b3 = fx_split(fx_shl(fx_mul(kFxA3, m), 2));
    return s;
}
// the multipliers times kappa, without rounding kappa times the scale to FP64
__host__ __device__ __forceinline__ fx_t fx_value(FxMul m) { return fx_shl((fx_t)m.h, 32) + m.l; }
__host__ __device__ __forceinline__ FxScale fx_scale_kappa(const FxScale& sc, double kap) {
    FxScale s;
    int ex;
    const FxMul m = fx_significand(kap, ex);
    const fx_t v0 = fx_mul(fx_value(sc.b0), m);
    const fx_t v1 = fx_mul(fx_value(sc.b1), m), v2 = fx_mul(fx_value(sc.b2), m), v3 = fx_mul(fx_value(sc.b3), m);
    const int l = v2 < (kFxA2 >> 3) ? 3 : 2;  // the product of the significands back to [1/2, 1)
    s.b0 = fx_split(fx_shl(v0, l));
    s.b1 = fx_split(fx_shl(v1, l));
    s.b2 = fx_split(fx_shl(v2, l));
    s.b3 = fx_split(fx_shl(v3, l));
    s.ex = sc.ex + ex + 2 - l;
    return s;
}

// A node value as a signed 53-bit significand (upper 54 bits) and an exponent
// field (lower 10): 0 for zero, 1 (and no significand) below 2^-422, kFxBad for
// what the fixed-point path leaves to FP64 (non-finite, 2^54 and above), else
// the biased exponent - 600.
constexpr int kFxTiny = -4000;  // exponent of a vanishing part
constexpr int kFxFp64 = 8000;   // marks contributions held as doubles
constexpr int kFxBias = 600, kFxBad = 1023, kFxMask = 1023;
constexpr int kFxMinExp = 1023 - 300 - kFxBias, kFxMaxExp = 1023 + 54 - kFxBias;
__host__ __device__ __forceinline__ fx_t fx_pack(double w) {
    const int hi = dbl_hi(w);
    const int be = (hi >> 20) & 0x7ff;
    const fx_t m = (dbl_bits(w) & 0xfffffffffffffLL) | 0x10000000000000LL;
    const fx_t sm = hi < 0 ? -m : m;
    int x = be - kFxBias;
    if (x >= kFxMaxExp) x = kFxBad;
    fx_t p = fx_shl(sm, 10) | x;
    if (x < 2) p = (dbl_bits(w) & 0x7fffffffffffffffLL) ? 1 : 0;
    return p;
}
__host__ __device__ __forceinline__ int fx_exp(fx_t p) { return (int)fx_lo(p) & kFxMask; }
// the largest exponent field of an element's corners: 0 for a zero element,
// which has zero contributions (0 x NaN and 0 x Inf apart); in range for fx_nd3 or not
__host__ __device__ __forceinline__ bool fx_exp_ok(int x) { return x >= kFxMinExp && x < kFxMaxExp; }
// a scale (node factor, kappa) fx_nd3 takes: in [2^-300, 2^300)
__host__ __device__ __forceinline__ bool fx_scale_ok(double scale) {
    const int h = dbl_hi(scale);  // (negative: sign bit set, fails the first test)
    return h >= ((1023 - 300) << 20) && h < ((1023 + 300) << 20);
}

// 2-point butterflies of element.cuh (exact here)
__host__ __device__ __forceinline__ void fx_h2_fwd(fx_t v00, fx_t v10, fx_t v01, fx_t v11, fx_t out[2][2]) {
    const fx_t t0p = v00 + v01, t0m = v00 - v01, t1p = v10 + v11, t1m = v10 - v11;
    out[1][1] = t0p + t1p;
    out[0][1] = t0p - t1p;
    out[1][0] = t0m + t1m;
    out[0][0] = t0m - t1m;
}
__host__ __device__ __forceinline__ void fx_h2_adj(const fx_t F[2][2], fx_t& w00, fx_t& w10, fx_t& w01, fx_t& w11) {
    const fx_t S0 = F[1][0] + F[0][0], S1 = F[1][1] + F[0][1];
    const fx_t D0 = F[1][0] - F[0][0], D1 = F[1][1] - F[0][1];
    w00 = S1 + S0;
    w01 = S1 - S0;
    w10 = D1 + D0;
    w11 = D1 - D0;
}

// Modes of an element's packed corner values p[8] with largest exponent field xm:
// W = w 2^k, M = T (x) T (x) T W; S = A^(p+q+r) M 2^(s-1) of the gradient modes, left-aligned
// by s (|M 2^s| < 2^62).
struct FxModes3 {
    fx_t M000, S001, S010, S100, S011, S101, S110, S111;
    int k, s;
};
__host__ __device__ __forceinline__ FxModes3 fx_modes3(const fx_t p[8], int xm) {
    FxModes3 m;
    m.k = 55 - (xm + kFxBias - 1022);
    fx_t u[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) u[c] = fx_sar(p[c] & ~(fx_t)kFxMask, 8 + xm - fx_exp(p[c]));
    const fx_t p0 = u[0] + u[1], q0 = u[1] - u[0], p1 = u[2] + u[3], q1 = u[3] - u[2];
    const fx_t p2 = u[4] + u[5], q2 = u[5] - u[4], p3 = u[6] + u[7], q3 = u[7] - u[6];
    const fx_t a00 = p0 + p1, a01 = p1 - p0, b00 = p2 + p3, b01 = p3 - p2;
    const fx_t a10 = q0 + q1, a11 = q1 - q0, b10 = q2 + q3, b11 = q3 - q2;
    m.M000 = a00 + b00;
    fx_t M[7] = {b00 - a00, a01 + b01, a10 + b10, b01 - a01, b10 - a10, a11 + b11, b11 - a11};
    // left-align the gradient modes: |M| < 2^(64 - clz), M' = M 2^s < 2^62
    unsigned int top = 0;
#pragma unroll
    for (int i = 0; i < 7; ++i) top |= (unsigned int)(fx_hi(M[i]) ^ (fx_hi(M[i]) >> 31));
    int s;
    if (top) {
        s = fx_clz(top) - 2;
    } else {  // differences below 2^-23 of the values: the bits are in the lower words
        unsigned int low = 0;
#pragma unroll
        for (int i = 0; i < 7; ++i) low |= fx_lo(M[i]) ^ (unsigned int)(fx_hi(M[i]) >> 31);
        s = 30 + fx_clz(low);
    }
    const FxMul A1 = fx_split(kFxA1), A2 = fx_split(kFxA2), A3 = fx_split(kFxA3);
    m.s = s;
    m.S001 = fx_mul(fx_shl(M[0], s), A1);
    m.S010 = fx_mul(fx_shl(M[1], s), A1);
    m.S100 = fx_mul(fx_shl(M[2], s), A1);
    m.S011 = fx_mul(fx_shl(M[3], s), A2);
    m.S101 = fx_mul(fx_shl(M[4], s), A2);
    m.S110 = fx_mul(fx_shl(M[5], s), A2);
    m.S111 = fx_mul(fx_shl(M[6], s), A3);
    return m;
}

// elem_nd3 (element.cuh) in fixed point: p[8] packed corner values with largest
// exponent field xm (fx_exp_ok), r[8] the contributions as integers times 2^X,
// the scale of `sc` applied.  Upper bounds: W 2^55, M 2^58, M' 2^62, S' 2^61,
// G 2^61.6, U 2^60, K 2^61, F 2^59.6, X 2^61.1, X+Y+Z 2^62.5, r 2^62.6.
__host__ __device__ __forceinline__ void fx_nd3(const fx_t p[8], int xm, const FxScale& sc, fx_t r[8], int& X) {
    const int e = xm + kFxBias - 1022;  // |w| < 2^e
    const FxModes3 m = fx_modes3(p, xm);
    const int k = m.k, s = m.s;
    fx_t P0[2][2], GX[2][2], GY[2][2], GZ[2][2];
    fx_h2_fwd(0, m.S010, m.S001, m.S011, P0);     // [sy][sz], without the constant mode
    fx_h2_fwd(m.S100, m.S110, m.S101, m.S111, GX);  // [sy][sz]
    fx_h2_fwd(m.S010, m.S110, m.S011, m.S111, GY);  // [sx][sz]
    fx_h2_fwd(m.S001, m.S101, m.S011, m.S111, GZ);  // [sx][sy]
    // 1 + u^2 at the points: U = u 2^(60 - max(e, 0)), K = (1 + u^2) 2^(60 - f)
    // with f = 2 max(e, 0); U carries 2^31 and K 2^30, so that the sum of two K
    // carries 2^31, which turns the lower words into rounded signed ones
    const int ep = e > 0 ? e : 0, f = 2 * ep;
    const fx_t one = (f > 60 ? 0 : (fx_t)1 << (60 - f)) + (fx_t)0x40000000LL;
    const fx_t U0 = fx_sar(fx_shl(m.M000, 2), ep - e) + (fx_t)0x80000000LL;
    const int shu = s - 3 + ep - e;
    fx_t K[2][2][2];
#pragma unroll
    for (int j = 0; j < 2; ++j)
#pragma unroll
        for (int l = 0; l < 2; ++l)
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const fx_t U = U0 + fx_sar(i ? P0[j][l] + GX[j][l] : P0[j][l] - GX[j][l], shu);
                const int uh = fx_hi(U) * 4, ul = (int)(fx_lo(U) ^ 0x80000000u);
                // (4 uh)^2 + 8 (4 uh ul / 2^32) = u^2 2^(60 - f)
                K[i][j][l] = one + ((fx_t)uh * uh + (fx_t)(fx_mulhi_s(uh, ul) * 2) * 4);
            }
    auto ksum = [](fx_t a, fx_t b) -> FxMul {
        const fx_t c = a + b;
        return {fx_hi(c), (int)(fx_lo(c) ^ 0x80000000u)};
    };
    fx_t FX[2][2], FY[2][2], FZ[2][2];
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            FX[i][j] = fx_mul(GX[i][j], ksum(K[1][i][j], K[0][i][j]));  // [sy][sz]
            FY[i][j] = fx_mul(GY[i][j], ksum(K[i][1][j], K[i][0][j]));  // [sx][sz]
            FZ[i][j] = fx_mul(GZ[i][j], ksum(K[i][j][1], K[i][j][0]));  // [sx][sy]
        }
    fx_t X00, X10, X01, X11, Y00, Y10, Y01, Y11, Z00, Z10, Z01, Z11;
    fx_h2_adj(FX, X00, X10, X01, X11);  // X_qr
    fx_h2_adj(FY, Y00, Y10, Y01, Y11);  // Y_pr
    fx_h2_adj(FZ, Z00, Z10, Z01, Z11);  // Z_pq
    const fx_t R100 = fx_mul(X00, sc.b1), R010 = fx_mul(Y00, sc.b1), R001 = fx_mul(Z00, sc.b1);
    const fx_t R110 = fx_mul(X10 + Y10, sc.b2), R101 = fx_mul(X01 + Z10, sc.b2), R011 = fx_mul(Y01 + Z01, sc.b2);
    const fx_t R111 = fx_mul(X11 + Y11 + Z11, sc.b3);
    const fx_t e01_0 = R010 - R011, e01_1 = R010 + R011, e10_0 = R100 - R101, e10_1 = R100 + R101;
    const fx_t e11_0 = R110 - R111, e11_1 = R110 + R111;
    const fx_t f0_00 = -R001 - e01_0, f0_10 = e01_0 - R001, f0_01 = R001 - e01_1, f0_11 = R001 + e01_1;
    const fx_t f1_00 = e10_0 - e11_0, f1_10 = e10_0 + e11_0, f1_01 = e10_1 - e11_1, f1_11 = e10_1 + e11_1;
    r[0] = f0_00 - f1_00; r[1] = f0_00 + f1_00;
    r[2] = f0_10 - f1_10; r[3] = f0_10 + f1_10;
    r[4] = f0_01 - f1_01; r[5] = f0_01 + f1_01;
    r[6] = f0_11 - f1_11; r[7] = f0_11 + f1_11;
    X = sc.ex + 3 + f - k - s;
}

// elem_vjp3 (element.cuh) in fixed point, without the coefficient's derivative:
// p[8] packed corner values of u with largest exponent field xu (below
// kFxMaxExp), q[8] of the covector w with xw (fx_exp_ok), r[8] times 2^X as above.
// The flux terms are those of fx_nd3 with the gradients of w; the source terms
// 2 u (grad u . grad w) have the exponent of a triple product, and the modes of
// both are summed at the larger of the two exponents.  Upper bounds: 4 dot
// 2^62.8, src 2^58.8, E 2^61.8, r 2^62.7.
__host__ __device__ __forceinline__ void fx_vjp3(const fx_t p[8], int xu, const fx_t q[8], int xw, const FxScale& sc,
                                                 fx_t r[8], int& X) {
    if (xu < kFxMinExp) xu = kFxMinExp;  // (u = 0, or so small that only 1 + u^2 = 1 is left of it)
    const int e = xu + kFxBias - 1022;
    const int ep = e > 0 ? e : 0, f = 2 * ep;
    const FxModes3 mw = fx_modes3(q, xw);
    fx_t G[2][2];
    FxMul WX[2][2], WY[2][2], WZ[2][2];
    auto split = [&](FxMul o[2][2]) {
#pragma unroll
        for (int c = 0; c < 4; ++c) o[c >> 1][c & 1] = fx_split(G[c >> 1][c & 1]);
    };
    fx_h2_fwd(mw.S100, mw.S110, mw.S101, mw.S111, G);  // [sy][sz]
    split(WX);
    fx_h2_fwd(mw.S010, mw.S110, mw.S011, mw.S111, G);  // [sx][sz]
    split(WY);
    fx_h2_fwd(mw.S001, mw.S101, mw.S011, mw.S111, G);  // [sx][sy]
    split(WZ);
    const FxModes3 mu = fx_modes3(p, xu);
    // u at the points (as in fx_nd3), and the three parts of grad u . grad w
    FxMul U[2][2][2];
    fx_t DX[2][2], DY[2][2], DZ[2][2];
    auto dots = [&](const FxMul w[2][2], fx_t o[2][2]) {
#pragma unroll
        for (int c = 0; c < 4; ++c) o[c >> 1][c & 1] = fx_mul(fx_split(G[c >> 1][c & 1]), w[c >> 1][c & 1]);
    };
    fx_h2_fwd(mu.S010, mu.S110, mu.S011, mu.S111, G);
    dots(WY, DY);
    fx_h2_fwd(mu.S001, mu.S101, mu.S011, mu.S111, G);
    dots(WZ, DZ);
    fx_h2_fwd(mu.S100, mu.S110, mu.S101, mu.S111, G);
    dots(WX, DX);
    {
        fx_t P0[2][2];
        fx_h2_fwd(0, mu.S010, mu.S001, mu.S011, P0);
        const fx_t U0 = fx_sar(fx_shl(mu.M000, 2), ep - e);
        const int shu = mu.s - 3 + ep - e;
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            const int i = c >> 2, j = c >> 1 & 1, l = c & 1;
            U[i][j][l] = fx_split(U0 + fx_sar(i ? P0[j][l] + G[j][l] : P0[j][l] - G[j][l], shu));
        }
    }
    const fx_t one = (f > 60 ? 0 : (fx_t)1 << (60 - f)) + (fx_t)0x40000000LL;  // (see fx_nd3)
    fx_t K[2][2][2], S[2][2][2];
#pragma unroll
    for (int c = 0; c < 8; ++c) {
        const int i = c >> 2, j = c >> 1 & 1, l = c & 1;
        const FxMul u = U[i][j][l];
        const int uh = u.h * 4;
        K[i][j][l] = one + ((fx_t)uh * uh + (fx_t)(fx_mulhi_s(uh, u.l) * 2) * 4);
        S[i][j][l] = fx_mul(fx_split(fx_shl(DX[j][l] + DY[i][l] + DZ[i][j], 2)), u);
    }
    auto ksum = [](fx_t a, fx_t b) -> FxMul {
        const fx_t c = a + b;
        return {fx_hi(c), (int)(fx_lo(c) ^ 0x80000000u)};
    };
    fx_t FX[2][2], FY[2][2], FZ[2][2], E0[2][2], E1[2][2];
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            FX[i][j] = fx_mul(WX[i][j], ksum(K[1][i][j], K[0][i][j]));  // [sy][sz]
            FY[i][j] = fx_mul(WY[i][j], ksum(K[i][1][j], K[i][0][j]));  // [sx][sz]
            FZ[i][j] = fx_mul(WZ[i][j], ksum(K[i][j][1], K[i][j][0]));  // [sx][sy]
            E0[i][j] = S[i][j][1] + S[i][j][0];
            E1[i][j] = S[i][j][1] - S[i][j][0];
        }
    fx_t X00, X10, X01, X11, Y00, Y10, Y01, Y11, Z00, Z10, Z01, Z11;
    fx_h2_adj(FX, X00, X10, X01, X11);  // X_qr
    fx_h2_adj(FY, Y00, Y10, Y01, Y11);  // Y_pr
    fx_h2_adj(FZ, Z00, Z10, Z01, Z11);  // Z_pq
    fx_t E000, E100, E010, E110, E001, E101, E011, E111;
    fx_h2_adj(E0, E000, E100, E010, E110);
    fx_h2_adj(E1, E001, E101, E011, E111);
    // exponents of the flux modes and of twice the source modes; the common one
    const int xf = 2 + f - mw.k - mw.s, xs = 63 + ep - mw.k - mw.s - mu.k - mu.s;
    const int xc = (xf > xs ? xf : xs) + 1;
    const int hf = xc - xf, hs = xc - xs;
    const fx_t R000 = fx_shl(fx_mul(fx_sar(E000, hs), sc.b0), 1);
    const fx_t R100 = fx_mul(fx_sar(X00, hf) + fx_sar(E100, hs), sc.b1);
    const fx_t R010 = fx_mul(fx_sar(Y00, hf) + fx_sar(E010, hs), sc.b1);
    const fx_t R001 = fx_mul(fx_sar(Z00, hf) + fx_sar(E001, hs), sc.b1);
    const fx_t R110 = fx_mul(fx_sar(X10 + Y10, hf) + fx_sar(E110, hs), sc.b2);
    const fx_t R101 = fx_mul(fx_sar(X01 + Z10, hf) + fx_sar(E101, hs), sc.b2);
    const fx_t R011 = fx_mul(fx_sar(Y01 + Z01, hf) + fx_sar(E011, hs), sc.b2);
    const fx_t R111 = fx_mul(fx_sar(X11 + Y11 + Z11, hf) + fx_sar(E111, hs), sc.b3);
    const fx_t e00_0 = R000 - R001, e00_1 = R000 + R001, e01_0 = R010 - R011, e01_1 = R010 + R011;
    const fx_t e10_0 = R100 - R101, e10_1 = R100 + R101, e11_0 = R110 - R111, e11_1 = R110 + R111;
    const fx_t f0_00 = e00_0 - e01_0, f0_10 = e00_0 + e01_0, f0_01 = e00_1 - e01_1, f0_11 = e00_1 + e01_1;
    const fx_t f1_00 = e10_0 - e11_0, f1_10 = e10_0 + e11_0, f1_01 = e10_1 - e11_1, f1_11 = e10_1 + e11_1;
    r[0] = f0_00 - f1_00; r[1] = f0_00 + f1_00;
    r[2] = f0_10 - f1_10; r[3] = f0_10 + f1_10;
    r[4] = f0_01 - f1_01; r[5] = f0_01 + f1_01;
    r[6] = f0_11 - f1_11; r[7] = f0_11 + f1_11;
    X = sc.ex + 1 + xc;
}

// ---------------------------------------------------------------------------
// 2D elements.  Corner index a + 2b; the three gradient modes are left-aligned
// as in 3D.
// ---------------------------------------------------------------------------
struct FxModes2 {
    fx_t m00, m10, m01, m11;  // m00 at 2^-k; the others at 2^-(k + s), below 2^62
    int k, s;
};
__host__ __device__ __forceinline__ FxModes2 fx_modes2(const fx_t p[4], int xm) {
    FxModes2 m;
    m.k = 55 - (xm + kFxBias - 1022);
    fx_t u[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) u[c] = fx_sar(p[c] & ~(fx_t)kFxMask, 8 + xm - fx_exp(p[c]));
    const fx_t p0 = u[0] + u[1], q0 = u[1] - u[0], p1 = u[2] + u[3], q1 = u[3] - u[2];
    m.m00 = p0 + p1;
    m.m10 = q0 + q1;
    m.m01 = p1 - p0;
    m.m11 = q1 - q0;
    auto mag = [](fx_t a) { return (unsigned int)(fx_hi(a) ^ (fx_hi(a) >> 31)); };
    const unsigned int top = mag(m.m10) | mag(m.m01) | mag(m.m11);
    if (top) {
        m.s = fx_clz(top) - 2;
    } else {
        auto low = [](fx_t a) { return fx_lo(a) ^ (unsigned int)(fx_hi(a) >> 31); };
        m.s = 30 + fx_clz(low(m.m10) | low(m.m01) | low(m.m11));
    }
    m.m10 = fx_shl(m.m10, m.s);
    m.m01 = fx_shl(m.m01, m.s);
    m.m11 = fx_shl(m.m11, m.s);
    return m;
}

// exp(U 2^-57) for |U| < 2^61: V 2^(N - 58), V in [2^58, 2^59].
//   exp(u) = 2^N 2^(j/256) exp(z), 256 N + j = floor(256 u / ln 2) (a little
//   below it at times), 0 <= z < 1.01 ln 2 / 256; exp(z) by its Taylor
//   polynomial of degree 5 (next term z^6 / 720 < 2^-60), the terms from z^3 on
//   in 32 bits (z^2 / 2 < 2^-18 times them).  Error below 2^-55 of exp(u).
__host__ __device__ __forceinline__ fx_t fx_exp_table(int j) {
#ifdef __CUDA_ARCH__
    return __ldg(&kFxExp2Dev[j]);
#else
    return kFxExp2Host[j];
#endif
}
__host__ __device__ __forceinline__ fx_t fx_exp(fx_t U, int& N) {
    const int n = (fx_mulhi_s(fx_hi(U), 1549082005) - 64) >> 15;  // 256 / ln 2 2^22; U's upper word is u 2^25
    // z 2^70: ln 2 / 256 2^70 = 0x2c5c85fdf473de6b
    const unsigned long long zs = ((unsigned long long)U << 13) - (unsigned long long)(long long)n * 0x2c5c85fdf473de6bULL;
    const unsigned int zh = (unsigned int)(zs >> 32), zl = (unsigned int)zs;   // zh = z 2^38
    const unsigned long long zz = (unsigned long long)zh * zh + 2ULL * fx_mulhi_u(zh, zl);  // z^2 2^76
    // S = z/3 + z^2/12 + z^3/60 = z (1/3 + z (1/12 + z/60))
    const unsigned int t1 = 1431655765u + fx_mulhi_u(zh, 4473924u);   // 1/12 + z/60, times 2^34
    const unsigned int t2 = 1431655765u + (fx_mulhi_u(zh, t1) >> 8);  // 1/3 + z t1, times 2^32
    const unsigned int S = (unsigned int)(((unsigned long long)zh * t2) >> 30);  // times 2^40
    // z^2/2 (1 + S): at 2^70
    const unsigned long long q = (zz >> 7) + (((unsigned long long)(unsigned int)(zz >> 27) * S) >> 20);
    // (1 + z + q) 2^61 times 2^(j/256) 2^61
    const fx_t F = ((fx_t)1 << 61) + (fx_t)((zs + q) >> 9);
    N = n >> 8;
    return fx_mul(F, fx_split(fx_exp_table(n & 255)));
}

// Source multipliers of the Bratu element: A^k |lh| 2^62 2^-ex, lh = lambda h^2 / 16.
struct FxBratu {
    FxMul b0, b1, b2;
    int ex;
    bool neg;
};
__host__ __device__ __forceinline__ FxBratu fx_bratu(double lh) {
    FxBratu s;
    s.neg = dbl_hi(lh) < 0;
    const double a = s.neg ? -lh : lh;
    if (a == 0.0) {
        s.b0 = s.b1 = s.b2 = FxMul{0, 0};
        s.ex = kFxTiny;
        return s;
    }
    s.b0 = fx_significand(a, s.ex);  // m 2^62
    s.b1 = fx_split(fx_shl(fx_mul(kFxA1, s.b0), 1));
    s.b2 = fx_split(fx_shl(fx_mul(kFxA2, s.b0), 1));
    return s;
}
__host__ __device__ __forceinline__ bool fx_bratu_ok(double lh) {
    return lh == 0.0 || fx_scale_ok(lh) || fx_scale_ok(-lh);
}
// elem_bratu2 takes |u| < 16
__host__ __device__ __forceinline__ bool fx_bratu_exp_ok(int x) { return x >= kFxMinExp && x < 1023 + 4 - kFxBias; }

// elem_bratu2 in fixed point; r[4] times 2^X, below 2^62.4
__host__ __device__ __forceinline__ void fx_bratu2(const fx_t p[4], int xm, const FxBratu& b, fx_t r[4], int& X) {
    const FxModes2 m = fx_modes2(p, xm);
    const FxMul A1 = fx_split(kFxA1), A2 = fx_split(kFxA2);
    // u at the points, times 2^57
    const fx_t T10 = fx_mul(m.m10, A1), T01 = fx_mul(m.m01, A1), T11 = fx_mul(m.m11, A2);
    const int e = 55 - m.k, sh = m.s - 1 - e;
    const fx_t U0 = e > 0 ? fx_shl(m.m00, e) : fx_sar(m.m00, -e);
    int N[4];
    fx_t V[4];
    V[0] = fx_exp(U0 + fx_sar(T11 - T10 - T01, sh), N[0]);   // (sx, sy) = (-, -)
    V[1] = fx_exp(U0 + fx_sar(T10 - T01 - T11, sh), N[1]);   // (+, -)
    V[2] = fx_exp(U0 + fx_sar(T01 - T10 - T11, sh), N[2]);   // (-, +)
    V[3] = fx_exp(U0 + fx_sar(T10 + T01 + T11, sh), N[3]);   // (+, +)
    const int n01 = N[0] > N[1] ? N[0] : N[1], n23 = N[2] > N[3] ? N[2] : N[3];
    const int nm = n01 > n23 ? n01 : n23;
#pragma unroll
    for (int q = 0; q < 4; ++q) V[q] = fx_sar(V[q], nm - N[q]);
    const fx_t s0 = V[0] + V[1], s1 = V[2] + V[3], d0 = V[1] - V[0], d1 = V[3] - V[2];
    // lh A^k E at 2^(nm + ex - 56)
    fx_t E00 = fx_mul(s1 + s0, b.b0), E01 = fx_mul(s1 - s0, b.b1), E10 = fx_mul(d1 + d0, b.b1), E11 = fx_mul(d1 - d0, b.b2);
    const int xs = nm + b.ex - 56, xg = -m.k - m.s - 1;
    X = (xs > xg ? xs : xg) + 1;
    const int ss = X - xs, sg = X - xg;
    const fx_t G10 = fx_sar(m.m10, sg + 1), G01 = fx_sar(m.m01, sg + 1), G11 = fx_sar(fx_mul(m.m11, fx_split(0x5555555555555555LL)), sg);
    E00 = fx_sar(E00, ss);
    E10 = fx_sar(E10, ss);
    E01 = fx_sar(E01, ss);
    E11 = fx_sar(E11, ss);
    const fx_t R00 = b.neg ? E00 : -E00;
    const fx_t R10 = b.neg ? G10 + E10 : G10 - E10;
    const fx_t R01 = b.neg ? G01 + E01 : G01 - E01;
    const fx_t R11 = b.neg ? G11 + E11 : G11 - E11;
    const fx_t g00 = R00 - R01, g01 = R00 + R01, g10 = R10 - R11, g11 = R10 + R11;
    r[0] = g00 - g10;
    r[1] = g00 + g10;
    r[2] = g01 - g11;
    r[3] = g01 + g11;
}

// 1 / sqrt(S 2^(F - 61)) times 2^61, for 0 < S < 2^62, F even and a result of at
// most 1: a 24-bit start from the hardware reciprocal square root and one
// third-order Newton step (error 5/16 e^3, e < 2^-21).
__host__ __device__ __forceinline__ fx_t fx_rsqrt(fx_t S, int F) {
    int n = fx_hi(S) ? fx_clz((unsigned int)fx_hi(S)) : 32 + fx_clz(fx_lo(S));
    n = (n - 3) | 1;  // odd, and m = S 2^n in [2^60, 2^62)
    const fx_t m = n > 0 ? fx_shl(S, n) : S >> 1;
    const float f = (float)fx_hi(m) * 0x1p-28f;  // m 2^-60 in [1, 4)
#ifdef __CUDA_ARCH__
    const unsigned int y0 = __float2uint_rn(rsqrtf(f) * 0x1p31f);
#else
    const unsigned int y0 = (unsigned int)std::lrint(1.0f / std::sqrt(f) * 0x1p31f);
#endif
    const fx_t e = ((fx_t)1 << 58) - fx_mul(m, fx_split((fx_t)((unsigned long long)y0 * y0)));  // (1 - m y0^2) 2^58
    const int e40 = (int)(e >> 18);
    const fx_t c4 = (e + ((fx_t)e40 * e40 * 3 >> 24)) * 8;  // (e/2 + 3/8 e^2) 2^62
    const fx_t y = fx_shl(y0, 30) + (fx_t)fx_hi(c4) * (fx_t)y0 + fx_mulhi_u(fx_lo(c4), y0);
    // S 2^(F - 61) = (m 2^-60) 2^(F - 1 - n)
    return fx_sar(y, (F - 1 - n) / 2);
}

// inv_h2 of the minimal-surface element, and the corner range it takes
struct FxMinsurf {
    FxMul m;
    int ex;
};
__host__ __device__ __forceinline__ FxMinsurf fx_minsurf(double inv_h2) {
    FxMinsurf s;
    s.m = fx_significand(inv_h2, s.ex);
    return s;
}
// elem_minsurf2 in fixed point; r[4] times 2^X, below 2^62.7.  False where a
// slope reaches 64 (left to FP64, as the coefficients then differ by more than
// their common scale should hold).
__host__ __device__ __forceinline__ bool fx_minsurf2(const fx_t p[4], int xm, const FxMinsurf& ih, fx_t r[4], int& X) {
    const FxModes2 m = fx_modes2(p, xm);
    const FxMul A1 = fx_split(kFxA1);
    // h grad u at 2^-(k + s)
    const fx_t gx0 = m.m10 >> 1, gy0 = m.m01 >> 1, gd = fx_mul(m.m11, A1);
    const fx_t gxm = gx0 - gd, gxp = gx0 + gd, gym = gy0 - gd, gyp = gy0 + gd;
    auto sq = [](fx_t g) -> fx_t {  // g^2 / 2^64
        const FxMul s = fx_split(g);
        return (fx_t)s.h * s.h + (fx_t)fx_mulhi_s(s.h, s.l) * 2;
    };
    const fx_t axm = sq(gxm), axp = sq(gxp), aym = sq(gym), ayp = sq(gyp);
    // (a + b) inv_h2 = p 2^xa, p < 2^59
    const int xa = ih.ex + 66 - 2 * (m.k + m.s);
    int F = xa + 59;
    if (F > 12) return false;
    F = F > 0 ? (F + 1) & ~1 : 0;
    const fx_t one = (fx_t)1 << (61 - F);
    const int sh = F - (xa + 59);
    auto coef = [&](fx_t a, fx_t b) -> fx_t { return fx_rsqrt(one + fx_sar(fx_shl(fx_mul(a + b, ih.m), 2), sh), F); };
    const fx_t cmm = coef(axm, aym), cpm = coef(axm, ayp), cmp = coef(axp, aym), cpp = coef(axp, ayp);
    const fx_t Xm = fx_mul(gxm, fx_split(cmm + cpm)), Xp = fx_mul(gxp, fx_split(cmp + cpp));
    const fx_t Ym = fx_mul(gym, fx_split(cmm + cmp)), Yp = fx_mul(gyp, fx_split(cpm + cpp));
    const fx_t P1 = Xm + Xp, P2 = Ym + Yp;
    const fx_t P3 = fx_shl(fx_mul((Xp - Xm) + (Yp - Ym), A1), 1);
    r[0] = P3 - P1 - P2;
    r[1] = P1 - P2 - P3;
    r[2] = P2 - P1 - P3;
    r[3] = P1 + P2 + P3;
    X = -m.k - m.s;
    return true;
}

// an integer times 2^X as a double (correctly rounded; X keeps it normal)
__host__ __device__ __forceinline__ double fx_to_double(fx_t a, int X) {
    const double d = fx_double(a);
    return dbl_hi(d) == 0 ? 0.0 : dbl_addexp(d, X * (1 << 20));
}

}  // namespace jfnk
