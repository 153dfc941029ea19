// 64-bit fixed-point evaluation of the 3D nonlinear-diffusion element, for the
// FP64 kernels.
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

// 1/sqrt 3, 1/3 and 1/(3 sqrt 3), times 2^63
constexpr fx_t kFxA1 = 0x49e69d1640cc7135LL, kFxA2 = 0x2aaaaaaaaaaaaaabLL, kFxA3 = 0x18a2345cc04425bcLL;

// Test-side multipliers of an element: A^k times a positive scale (the node
// factor, and kappa), its power of two apart.  b_k = A^k m 2^63, scale = m 2^ex
// with m in [1/2, 1).
struct FxScale {
    FxMul b1, b2, b3;
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
    const fx_t v1 = fx_mul(fx_value(sc.b1), m), v2 = fx_mul(fx_value(sc.b2), m), v3 = fx_mul(fx_value(sc.b3), m);
    const int l = v2 < (kFxA2 >> 3) ? 3 : 2;  // the product of the significands back to [1/2, 1)
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
// which has zero contributions; in range for fx_nd3 or not
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

// elem_nd3 (element.cuh) in fixed point: p[8] packed corner values with largest
// exponent field xm (fx_exp_ok), r[8] the contributions as integers times 2^X,
// the scale of `sc` applied.  Upper bounds: W 2^55, M 2^58, M' 2^62, S' 2^61,
// G 2^61.6, U 2^60, K 2^61, F 2^59.6, X 2^61.1, X+Y+Z 2^62.5, r 2^62.6.
__host__ __device__ __forceinline__ void fx_nd3(const fx_t p[8], int xm, const FxScale& sc, fx_t r[8], int& X) {
    const int e = xm + kFxBias - 1022;  // |w| < 2^e
    const int k = 55 - e;               // W = w 2^k
    fx_t u[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) u[c] = fx_sar(p[c] & ~(fx_t)kFxMask, 8 + xm - fx_exp(p[c]));
    // modes (as in elem_nd3)
    const fx_t p0 = u[0] + u[1], q0 = u[1] - u[0], p1 = u[2] + u[3], q1 = u[3] - u[2];
    const fx_t p2 = u[4] + u[5], q2 = u[5] - u[4], p3 = u[6] + u[7], q3 = u[7] - u[6];
    const fx_t a00 = p0 + p1, a01 = p1 - p0, b00 = p2 + p3, b01 = p3 - p2;
    const fx_t a10 = q0 + q1, a11 = q1 - q0, b10 = q2 + q3, b11 = q3 - q2;
    const fx_t M000 = a00 + b00;
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
    const fx_t S001 = fx_mul(fx_shl(M[0], s), A1), S010 = fx_mul(fx_shl(M[1], s), A1), S100 = fx_mul(fx_shl(M[2], s), A1);
    const fx_t S011 = fx_mul(fx_shl(M[3], s), A2), S101 = fx_mul(fx_shl(M[4], s), A2), S110 = fx_mul(fx_shl(M[5], s), A2);
    const fx_t S111 = fx_mul(fx_shl(M[6], s), A3);
    fx_t P0[2][2], GX[2][2], GY[2][2], GZ[2][2];
    fx_h2_fwd(0, S010, S001, S011, P0);     // [sy][sz], without the constant mode
    fx_h2_fwd(S100, S110, S101, S111, GX);  // [sy][sz]
    fx_h2_fwd(S010, S110, S011, S111, GY);  // [sx][sz]
    fx_h2_fwd(S001, S101, S011, S111, GZ);  // [sx][sy]
    // 1 + u^2 at the points: U = u 2^(60 - max(e, 0)), K = (1 + u^2) 2^(60 - f)
    // with f = 2 max(e, 0); U carries 2^31 and K 2^30, so that the sum of two K
    // carries 2^31, which turns the lower words into rounded signed ones
    const int ep = e > 0 ? e : 0, f = 2 * ep;
    const fx_t one = (f > 60 ? 0 : (fx_t)1 << (60 - f)) + (fx_t)0x40000000LL;
    const fx_t U0 = fx_sar(fx_shl(M000, 2), ep - e) + (fx_t)0x80000000LL;
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

// an integer times 2^X as a double (correctly rounded; X keeps it normal)
__host__ __device__ __forceinline__ double fx_to_double(fx_t a, int X) {
    const double d = fx_double(a);
    return dbl_hi(d) == 0 ? 0.0 : dbl_addexp(d, X * (1 << 20));
}

}  // namespace jfnk
