// Neo-Hookean hexahedron of the beam in FP64: elem_neohooke (element.cuh),
// factorised.
//
// elem_neohooke evaluates every Gauss point's gradient from the 8 corners and
// scatters every point's stress to them, about 2400 FP64 operations, and the
// FP64 pipe (2 a clock and SM) bounds it.  Here the corner values become
// gradients at the points, and the stresses corner contributions, by the x, y
// and z butterflies of the scalar elements, in 64-bit fixed point (fx64.cuh);
// ln J and 1 / J come from fixed point too.  What is left on the FP64 pipe is
// the stress itself: 39 operations a point, and 12 conversions a component and
// side.  Residual on 160 x 16 x 16 elements 350 -> 71 us (element kernel and node
// kernel).
#pragma once
#include "element.cuh"
#include "fx64.cuh"

namespace jfnk {

#ifdef __CUDACC__
static __device__ const short kFxLogCDev[128] = {JFNK_FX_LOG_C};
static __device__ const fx_t kFxLogLDev[128] = {JFNK_FX_LOG_L};
#endif
static const short kFxLogCHost[128] = {JFNK_FX_LOG_C};
static const fx_t kFxLogLHost[128] = {JFNK_FX_LOG_L};

// ln x 2^57 (error below 2^-54) and 1 / x (below 2^-52 of it) for 2^-16 <= x < 2^16; false outside.
//   x = 2^j m: with c from a table of 128 intervals, r = m c / 1024 - 1 (exact,
//   |r| < 2^-7.6) and ln m = l + ln(1 + r), the logarithm's series to r^7, from
//   r^3 on in 32 bits.  1 / m: a 24-bit start from FP32 and one third-order step.
__host__ __device__ __forceinline__ bool fx_log_rcp(double x, fx_t& ln, double& rcp) {
    const int hi = dbl_hi(x);
    if (hi < ((1023 - 16) << 20) || hi >= ((1023 + 16) << 20)) return false;  // (negative, NaN too)
    const int j = (hi >> 20) - 1023;
    const fx_t m = (dbl_bits(x) & 0xfffffffffffffLL) | 0x10000000000000LL;  // m 2^52
    const int i = (hi >> 13) & 127;
#ifdef __CUDA_ARCH__
    const int c = __ldg(&kFxLogCDev[i]);
    const fx_t l = __ldg(&kFxLogLDev[i]);
#else
    const int c = kFxLogCHost[i];
    const fx_t l = kFxLogLHost[i];
#endif
    const fx_t r = m * c - ((fx_t)1 << 62);  // r 2^62
    const int rh = (int)(r >> 24);           // r 2^38, below 2^31
    // r^2 2^64 (r 2^62 = rs: its split product with itself, times 2^4)
    const FxMul rs = fx_split(fx_shl(r, 4));  // r 2^66, below 2^59
    const fx_t r2 = (fx_t)rs.h * rs.h + (fx_t)fx_mulhi_s(rs.h, rs.l) * 2;  // r^2 2^68
    // Q = -1/2 + r U, U = 1/3 + r V, V = -1/4 + r (1/5 + r (-1/6 + r/7))
    const int v3 = -715827883 + (fx_mulhi_s(rh, 613566757) >> 6);  // -1/6 + r/7, times 2^32
    const int v2 = 858993459 + (fx_mulhi_s(rh, v3) >> 6);          // 1/5 + ..., times 2^32
    const int V = -1073741824 + (fx_mulhi_s(rh, v2) >> 6);         // times 2^32
    const fx_t U = 366503875925LL + (((fx_t)rh * V) >> 30);        // times 2^40
    const fx_t Q = -((fx_t)1 << 59) + fx_mul(fx_shl(r, 1), fx_split(fx_shl(U, 21)));  // U 2^61: times 2^60
    // r2 is positive and below 2^53: ln(1 + r) 2^57 = r 2^57 + r^2 Q 2^57
    ln = (r >> 5) + (fx_mul(Q, fx_split(fx_shl(r2, 8))) >> 15) + l + (fx_t)j * 0x162e42fefa39ef3LL;
    // 1 / m in (1/2, 1]: m 2^61 times y0 2^31
    const float f = (float)(int)(m >> 22) * 0x1p-30f;
    const unsigned int y0 = (unsigned int)(1.0f / f * 0x1p31f);
    const fx_t e = ((fx_t)1 << 58) - fx_mul(fx_shl(m, 9), fx_split(fx_shl(y0, 30)));  // (1 - m y0) 2^58
    const int e40 = (int)(e >> 18);
    const fx_t c4 = (e + ((fx_t)e40 * e40 >> 22)) * 16;  // (e + e^2) 2^62
    const fx_t y = fx_shl(y0, 30) + (fx_t)fx_hi(c4) * (fx_t)y0 + fx_mulhi_u(fx_lo(c4), y0);  // times 2^61
    rcp = dbl_addexp(fx_double(y), (-61 - j) * (1 << 20));
    return true;
}

struct FxBeam {
    FxMul f0, f1, f2;  // A^k times inv_h / 4, times 2^62 2^-fe
    FxMul b0, b1, b2;  // A^k times h^2 / 32
    int fe, be;
};
__host__ __device__ __forceinline__ void fx_beam_mul(double scale, FxMul& m0, FxMul& m1, FxMul& m2, int& e) {
    m0 = fx_significand(scale, e);
    m1 = fx_split(fx_shl(fx_mul(kFxA1, m0), 1));
    m2 = fx_split(fx_shl(fx_mul(kFxA2, m0), 1));
}
__host__ __device__ __forceinline__ FxBeam fx_beam(double inv_h) {
    FxBeam b;
    const double h = 1.0 / inv_h;
    fx_beam_mul(0.25 * inv_h, b.f0, b.f1, b.f2, b.fe);
    fx_beam_mul(0.03125 * h * h, b.b0, b.b1, b.b2, b.be);
    return b;
}

// elem_neohooke's r for u; false where a value leaves the ranges above.
__host__ __device__ __forceinline__ bool fx_neohooke(const double u[24], const FxBeam& b, double r[24]) {
    // displacement gradients: GX[i] at [sy][sz], GY[i] at [sx][sz], GZ[i] at [sx][sy]
    double GX[3][2][2], GY[3][2][2], GZ[3][2][2];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        fx_t p[8], w[8];
        int xm = 0;
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            p[c] = fx_pack(u[3 * c + i]);
            xm = fx_exp(p[c]) > xm ? fx_exp(p[c]) : xm;
        }
        if (xm != 0 && !fx_exp_ok(xm)) return false;
        const int k = 55 - (xm + kFxBias - 1022);
#pragma unroll
        for (int c = 0; c < 8; ++c) w[c] = fx_sar(p[c] & ~(fx_t)kFxMask, 8 + xm - fx_exp(p[c]));
        const fx_t p0 = w[0] + w[1], q0 = w[1] - w[0], p1 = w[2] + w[3], q1 = w[3] - w[2];
        const fx_t p2 = w[4] + w[5], q2 = w[5] - w[4], p3 = w[6] + w[7], q3 = w[7] - w[6];
        const fx_t a00 = p0 + p1, a01 = p1 - p0, b00 = p2 + p3, b01 = p3 - p2;
        const fx_t a10 = q0 + q1, a11 = q1 - q0, b10 = q2 + q3, b11 = q3 - q2;
        const fx_t M[7] = {b00 - a00, a01 + b01, a10 + b10, b01 - a01, b10 - a10, a11 + b11, b11 - a11};
        unsigned int top = 0, low = 0;
#pragma unroll
        for (int q = 0; q < 7; ++q) {
            top |= (unsigned int)(fx_hi(M[q]) ^ (fx_hi(M[q]) >> 31));
            low |= fx_lo(M[q]) ^ (unsigned int)(fx_hi(M[q]) >> 31);
        }
        const int s = top ? fx_clz(top) - 2 : 30 + fx_clz(low);
        const fx_t S001 = fx_mul(fx_shl(M[0], s), b.f0), S010 = fx_mul(fx_shl(M[1], s), b.f0);
        const fx_t S100 = fx_mul(fx_shl(M[2], s), b.f0), S011 = fx_mul(fx_shl(M[3], s), b.f1);
        const fx_t S101 = fx_mul(fx_shl(M[4], s), b.f1), S110 = fx_mul(fx_shl(M[5], s), b.f1);
        const fx_t S111 = fx_mul(fx_shl(M[6], s), b.f2);
        const int X = 2 - k - s + b.fe;
        fx_t g[2][2];
        fx_h2_fwd(S100, S110, S101, S111, g);
#pragma unroll
        for (int q = 0; q < 4; ++q) GX[i][q >> 1][q & 1] = fx_to_double(g[q >> 1][q & 1], X);
        fx_h2_fwd(S010, S110, S011, S111, g);
#pragma unroll
        for (int q = 0; q < 4; ++q) GY[i][q >> 1][q & 1] = fx_to_double(g[q >> 1][q & 1], X);
        fx_h2_fwd(S001, S101, S011, S111, g);
#pragma unroll
        for (int q = 0; q < 4; ++q) GZ[i][q >> 1][q & 1] = fx_to_double(g[q >> 1][q & 1], X);
        double (&D)[2][2] = i == 0 ? GX[0] : i == 1 ? GY[1] : GZ[2];  // F = I + grad u
#pragma unroll
        for (int q = 0; q < 4; ++q) D[q >> 1][q & 1] += 1.0;
    }
    // stress at the points, summed over the direction its test gradient does not
    // depend on: FX[i] at [sy][sz], FY[i] at [sx][sz], FZ[i] at [sx][sy]
    double FX[3][2][2], FY[3][2][2], FZ[3][2][2];
    bool ok = true;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        const int sx = q & 1, sy = (q >> 1) & 1, sz = q >> 2;
        const double F00 = GX[0][sy][sz], F01 = GY[0][sx][sz], F02 = GZ[0][sx][sy];
        const double F10 = GX[1][sy][sz], F11 = GY[1][sx][sz], F12 = GZ[1][sx][sy];
        const double F20 = GX[2][sy][sz], F21 = GY[2][sx][sz], F22 = GZ[2][sx][sy];
        const double C00 = F11 * F22 - F12 * F21, C01 = F12 * F20 - F10 * F22, C02 = F10 * F21 - F11 * F20;
        const double C10 = F02 * F21 - F01 * F22, C11 = F00 * F22 - F02 * F20, C12 = F01 * F20 - F00 * F21;
        const double C20 = F01 * F12 - F02 * F11, C21 = F02 * F10 - F00 * F12, C22 = F00 * F11 - F01 * F10;
        const double J = F00 * C00 + F01 * C01 + F02 * C02;
        fx_t ln = 0;
        double rJ = 0.0;
        ok = fx_log_rcp(J, ln, rJ) && ok;
        const double kc = (kBeamLambda * fx_to_double(ln, -57) - kBeamMu) * rJ;
        auto add = [&](double& acc, double F, double C, bool first) {
            acc = first ? kc * C + kBeamMu * F : kc * C + (kBeamMu * F + acc);
        };
        add(FX[0][sy][sz], F00, C00, sx == 0);
        add(FY[0][sx][sz], F01, C01, sy == 0);
        add(FZ[0][sx][sy], F02, C02, sz == 0);
        add(FX[1][sy][sz], F10, C10, sx == 0);
        add(FY[1][sx][sz], F11, C11, sy == 0);
        add(FZ[1][sx][sy], F12, C12, sz == 0);
        add(FX[2][sy][sz], F20, C20, sx == 0);
        add(FY[2][sx][sz], F21, C21, sy == 0);
        add(FZ[2][sx][sy], F22, C22, sz == 0);
    }
    if (!ok) return false;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        fx_t p[12];
        int xm = 0;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            p[q] = fx_pack(FX[i][q >> 1][q & 1]);
            p[4 + q] = fx_pack(FY[i][q >> 1][q & 1]);
            p[8 + q] = fx_pack(FZ[i][q >> 1][q & 1]);
        }
#pragma unroll
        for (int q = 0; q < 12; ++q) xm = fx_exp(p[q]) > xm ? fx_exp(p[q]) : xm;
        if (xm == 0) {
#pragma unroll
            for (int c = 0; c < 8; ++c) r[3 * c + i] = 0.0;
            continue;
        }
        if (!fx_exp_ok(xm)) return false;
        // W = F 2^(59 - e), |F| < 2^e
        fx_t W[12];
#pragma unroll
        for (int q = 0; q < 12; ++q) W[q] = fx_sar(p[q] & ~(fx_t)kFxMask, 4 + xm - fx_exp(p[q]));
        fx_t g[2][2], X00, X10, X01, X11, Y00, Y10, Y01, Y11, Z00, Z10, Z01, Z11;
#pragma unroll
        for (int q = 0; q < 4; ++q) g[q >> 1][q & 1] = W[q];
        fx_h2_adj(g, X00, X10, X01, X11);
#pragma unroll
        for (int q = 0; q < 4; ++q) g[q >> 1][q & 1] = W[4 + q];
        fx_h2_adj(g, Y00, Y10, Y01, Y11);
#pragma unroll
        for (int q = 0; q < 4; ++q) g[q >> 1][q & 1] = W[8 + q];
        fx_h2_adj(g, Z00, Z10, Z01, Z11);
        const fx_t R100 = fx_mul(X00, b.b0), R010 = fx_mul(Y00, b.b0), R001 = fx_mul(Z00, b.b0);
        const fx_t R110 = fx_mul(X10 + Y10, b.b1), R101 = fx_mul(X01 + Z10, b.b1), R011 = fx_mul(Y01 + Z01, b.b1);
        const fx_t R111 = fx_mul(X11 + Y11 + Z11, b.b2);
        const int X = 2 - (59 - (xm + kFxBias - 1022)) + b.be;
        const fx_t e01_0 = R010 - R011, e01_1 = R010 + R011, e10_0 = R100 - R101, e10_1 = R100 + R101;
        const fx_t e11_0 = R110 - R111, e11_1 = R110 + R111;
        const fx_t f0_00 = -R001 - e01_0, f0_10 = e01_0 - R001, f0_01 = R001 - e01_1, f0_11 = R001 + e01_1;
        const fx_t f1_00 = e10_0 - e11_0, f1_10 = e10_0 + e11_0, f1_01 = e10_1 - e11_1, f1_11 = e10_1 + e11_1;
        r[i] = fx_to_double(f0_00 - f1_00, X);
        r[3 + i] = fx_to_double(f0_00 + f1_00, X);
        r[6 + i] = fx_to_double(f0_10 - f1_10, X);
        r[9 + i] = fx_to_double(f0_10 + f1_10, X);
        r[12 + i] = fx_to_double(f0_01 - f1_01, X);
        r[15 + i] = fx_to_double(f0_01 + f1_01, X);
        r[18 + i] = fx_to_double(f0_11 - f1_11, X);
        r[21 + i] = fx_to_double(f0_11 + f1_11, X);
    }
    return true;
}

}  // namespace jfnk
