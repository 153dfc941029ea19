// Host check of the fixed-point element (csrc/fx64.cuh) against the FP64 one
// (csrc/element.cuh), both against a long double quadrature.  Built with
// -fsanitize=signed-integer-overflow, so an intermediate that leaves its 64 (or
// 32) bits ends the program.
//   1. single elements: every sign pattern of the 8 corners, exponents over the
//      accepted range, corners of equal and of very different size, kappa over
//      its range.  Worst case of the bit budget: 2^7 units on a largest
//      contribution of at least 2^54, i.e. 2^-47 of it.
//   2. the 2D elements likewise.
//   3. fields assembled over 6^3 elements: the error's 2-norm is at most 1.5
//      times that of the FP64 element (a quarter to a hundredth where the
//      field is smooth or random).
// Prints violations and "ok <cases>".
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <random>
#include <vector>

#include "element.cuh"
#include "fx64.cuh"

using namespace jfnk;
typedef long double Q;

static void reference(const double w[8], Q kap, Q r[8]) {
    const Q a = 1 / (2 * std::sqrt((Q)3));
    for (int c = 0; c < 8; ++c) r[c] = 0;
    for (int q = 0; q < 8; ++q) {
        Q N[8], G[8][3], u = 0, g[3] = {0, 0, 0};
        for (int c = 0; c < 8; ++c) {
            Q l[3], s[3];
            for (int d = 0; d < 3; ++d) {
                const Q p = (q >> d & 1) ? (Q)0.5 + a : (Q)0.5 - a;
                l[d] = (c >> d & 1) ? p : 1 - p;
                s[d] = (c >> d & 1) ? 1 : -1;
            }
            N[c] = l[0] * l[1] * l[2];
            G[c][0] = s[0] * l[1] * l[2];
            G[c][1] = s[1] * l[0] * l[2];
            G[c][2] = s[2] * l[0] * l[1];
            u += N[c] * w[c];
            for (int d = 0; d < 3; ++d) g[d] += G[c][d] * w[c];
        }
        const Q k = kap * (1 + u * u) / 8 * 16 / 3;  // contributions over 3 h / 16, as elem_nd3
        for (int c = 0; c < 8; ++c)
            for (int d = 0; d < 3; ++d) r[c] += k * g[d] * G[c][d];
    }
}

// contributions times `scale`; false where the element is left to FP64
static bool fixed(const double w[8], double kap, double scale, double r[8]) {
    fx_t p[8], ri[8];
    int xm = 0, X = 0;
    for (int c = 0; c < 8; ++c) {
        p[c] = fx_pack(w[c]);
        xm = std::max(xm, fx_exp(p[c]));
    }
    if (!fx_exp_ok(xm) || !fx_scale_ok(kap)) return false;
    fx_nd3(p, xm, kap == 1.0 ? fx_scale(scale) : fx_scale_kappa(fx_scale(scale), kap), ri, X);
    for (int c = 0; c < 8; ++c) r[c] = fx_to_double(ri[c], X);
    return true;
}

static std::mt19937_64 rng(11);
static double uni() { return std::uniform_real_distribution<double>(-1, 1)(rng); }
static double nrm() { return std::normal_distribution<double>()(rng); }

// 2D elements: Bratu (par = lambda h^2 / 16) or minimal surface (par = 1 / h^2)
static void reference2(bool ms, const double w[4], Q par, Q r[4]) {
    const Q a = 1 / (2 * std::sqrt((Q)3));
    for (int c = 0; c < 4; ++c) r[c] = 0;
    for (int q = 0; q < 4; ++q) {
        const Q px = (q & 1) ? (Q)0.5 + a : (Q)0.5 - a, py = (q & 2) ? (Q)0.5 + a : (Q)0.5 - a;
        Q N[4], gx[4], gy[4], u = 0, x = 0, y = 0;
        for (int c = 0; c < 4; ++c) {
            const Q lx = (c & 1) ? px : 1 - px, ly = (c & 2) ? py : 1 - py;
            N[c] = lx * ly;
            gx[c] = (c & 1) ? ly : -ly;
            gy[c] = (c & 2) ? lx : -lx;
            u += N[c] * w[c];
            x += gx[c] * ((Q)w[c] - w[0]);  // (the gradients' weights sum to zero)
            y += gy[c] * ((Q)w[c] - w[0]);
        }
        const Q k = ms ? 1 / std::sqrt(1 + (x * x + y * y) * par) : (Q)1;
        for (int c = 0; c < 4; ++c) {
            r[c] += k * (x * gx[c] + y * gy[c]) / 4;
            if (!ms) r[c] -= 4 * par * std::exp(u) * N[c];
        }
    }
}

// single 2D elements: errors against the element's largest contribution or
// source.  Bit budget: 2^6 units on at least 2^55 (exp 2^-55, rsqrt 2^-54).
static int check2(int& cases) {
    int bad = 0;
    for (int ms = 0; ms < 2; ++ms)
        for (int ex : {-290, -100, -30, -6, -1, 0, 1, 3})
            for (int it = 0; it < 400; ++it) {
                const double par = ms ? std::ldexp(1.0 + std::fabs(uni()), (it % 4 == 0 ? 12 : 3) - 2 * ex)
                                      : (it % 7 ? 1 : -1) * std::ldexp(std::fabs(uni()), -(int)(rng() % 30));
                double w[4];
                fx_t p[4], r[4];
                int xm = 0, X = 0;
                for (int c = 0; c < 4; ++c) {
                    w[c] = std::ldexp(it % 3 == 0 ? uni() : it % 3 == 1 ? ((it >> (c + 2)) & 1 ? 0.999 : -0.999) : 0.7 + 1e-10 * uni(), ex);
                    p[c] = fx_pack(w[c]);
                    xm = std::max(xm, fx_exp(p[c]));
                }
                ++cases;
                Q q[4], big = 0, err = 0;
                reference2(ms, w, par, q);
                if (ms) {
                    if (!fx_exp_ok(xm) || !fx_minsurf2(p, xm, fx_minsurf(par), r, X)) continue;  // left to FP64
                } else {
                    if (!fx_exp_ok(xm) || !fx_bratu_exp_ok(xm)) { printf("2D refused: %d\n", ex), ++bad; continue; }
                    fx_bratu2(p, xm, fx_bratu(par), r, X);
                    big = std::fabs((Q)par) * std::exp((Q)std::max({w[0], w[1], w[2], w[3]}));
                }
                for (int c = 0; c < 4; ++c) {
                    big = std::max(big, std::fabs(q[c]));
                    err = std::max(err, std::fabs(q[c] - (Q)fx_to_double(r[c], X)));
                }
                if (!(err <= 0x1p-49L * big)) printf("2D %d exponent %d case %d: %Lg of %Lg\n", ms, ex, it, err, big), ++bad;
            }
    return bad;
}

int main() {
    int bad = 0, cases = 0;
    bad += check2(cases);
    const double scale = 3.0 / 16 / 100;
    const int exps[] = {-299, -120, -40, -8, -2, -1, 0, 1, 2, 9, 30, 53};
    for (int ex : exps)
        for (int size = 0; size < 5; ++size)
            for (int sign = 0; sign < 256; ++sign) {
                double w[8], r[8];
                const double kap = size == 4 ? std::exp(60 * uni()) : 1.0;
                for (int c = 0; c < 8; ++c) {
                    const double m = size == 0 ? 1 - 0x1p-53 : size == 1 ? 0.5 + 0.5 * std::fabs(uni())
                                     : size == 2 ? std::ldexp(1.0, -(int)(rng() % 40)) * 0.999
                                     : size == 3 ? 1 - 1e-11 * std::fabs(uni()) : std::fabs(uni());
                    w[c] = std::ldexp((sign >> c & 1) ? -m : m, ex);
                }
                w[sign & 7] = std::ldexp(w[sign & 7] < 0 ? -0.75 : 0.75, ex);
                Q q[8], big = 0, err = 0;
                reference(w, (Q)kap * scale, q);
                ++cases;
                if (!fixed(w, kap, scale, r)) {
                    printf("refused: exponent %d size %d\n", ex, size), ++bad;
                    continue;
                }
                for (int c = 0; c < 8; ++c) {
                    big = std::max(big, std::fabs(q[c]));
                    err = std::max(err, std::fabs(q[c] - r[c]));
                }
                if (!(err <= 0x1p-47L * big)) printf("exponent %d size %d sign %d: %Lg of %Lg\n", ex, size, sign, err, big), ++bad;
            }
    // left to FP64
    const double out[] = {INFINITY, -INFINITY, NAN, 0x1p54, -1e300, 1e-100, 4e-320};
    for (double x : out) {
        double w[8] = {0, 0, 0, x, 0, 0, 0, 0}, r[8];
        ++cases;
        if (fixed(w, 1.0, scale, r)) printf("taken: %g\n", x), ++bad;
        if (fx_exp(fx_pack(x)) == 0) printf("packed as zero: %g\n", x), ++bad;
    }
    const double kout[] = {0.0, -0.0, -1.0, INFINITY, NAN, 1e-100, 1e100};
    for (double k : kout) {
        double w[8] = {1, 1, 1, 1, 1, 1, 1, 0}, r[8];
        ++cases;
        if (fixed(w, k, scale, r)) printf("kappa taken: %g\n", k), ++bad;
    }
    // assembled fields
    const int m = 6;
    for (int kind = 0; kind < 9; ++kind)
        for (int kp = 0; kp < 2; ++kp) {
            Q e64 = 0, efx = 0;
            for (int trial = 0; trial < 30; ++trial) {
                const int n = kind == 0 ? 16 : kind == 1 ? 64 : kind == 2 ? 256 : 128;
                double o[3];
                for (double& x : o) x = 0.5 * (uni() + 1) * (1 - m / (double)n);
                std::vector<double> w((m + 1) * (m + 1) * (m + 1));
                auto id = [&](int x, int y, int z) { return (z * (m + 1) + y) * (m + 1) + x; };
                for (int z = 0; z <= m; ++z)
                    for (int y = 0; y <= m; ++y)
                        for (int x = 0; x <= m; ++x) {
                            const double s = std::sin(M_PI * (o[0] + x / (double)n)) * std::sin(M_PI * (o[1] + y / (double)n)) *
                                             std::sin(M_PI * (o[2] + z / (double)n));
                            const double v[] = {s, s, s, s + 0.1 * nrm(), uni(), 1e-8 * s, 1e3 * s, 1 + 1e-9 * nrm(), 1e-30 * nrm()};
                            w[id(x, y, z)] = v[kind];
                        }
                std::vector<Q> R(w.size(), 0);
                std::vector<double> A(w.size(), 0), B(w.size(), 0);
                for (int z = 0; z < m; ++z)
                    for (int y = 0; y < m; ++y)
                        for (int x = 0; x < m; ++x) {
                            double u[8], a[8], b[8];
                            Q q[8];
                            for (int c = 0; c < 8; ++c) u[c] = w[id(x + (c & 1), y + (c >> 1 & 1), z + (c >> 2))];
                            const double kap = kp ? std::exp(0.7 * nrm()) : 1.0;
                            reference(u, (Q)kap * scale, q);
                            if (kp) elem_nd3<double, true>(u, kap, a);
                            else elem_nd3<double, false>(u, 1.0, a);
                            if (!fixed(u, kap, scale, b)) printf("refused: field %d\n", kind), ++bad;
                            for (int c = 0; c < 8; ++c) {
                                const int i = id(x + (c & 1), y + (c >> 1 & 1), z + (c >> 2));
                                R[i] += q[c];
                                A[i] += a[c];
                                B[i] += b[c];
                            }
                        }
                for (int z = 1; z < m; ++z)
                    for (int y = 1; y < m; ++y)
                        for (int x = 1; x < m; ++x) {
                            const int i = id(x, y, z);
                            e64 += (A[i] * scale - R[i]) * (A[i] * scale - R[i]);
                            efx += (B[i] - R[i]) * (B[i] - R[i]);
                        }
            }
            ++cases;
            if (!(efx <= 1.5L * 1.5L * e64)) printf("field %d kappa %d: %Lg against %Lg\n", kind, kp, std::sqrt(efx), std::sqrt(e64)), ++bad;
        }
    if (!bad) printf("ok %d\n", cases);
    return bad != 0;
}
