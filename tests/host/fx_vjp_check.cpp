// Host check of the fixed-point vector-Jacobian product (csrc/fx64.cuh:
// fx_vjp3) against the FP64 one (csrc/element.cuh: elem_vjp3), both against a
// long double quadrature.  Built with -fsanitize=signed-integer-overflow.
//   1. single elements: sign patterns and exponents of u and of the covector
//      over the accepted ranges.  Error budget: 2^7 units of the contributions,
//      whose flux part is kept to up to 3 bits less than in the residual where the
//      source part needs the room: 2^-44 of the sum of the terms' magnitudes.
//   2. fields assembled over 5^3 elements: the error's 2-norm is at most 1.5
//      times that of the FP64 element.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <random>
#include <vector>

#include "element.cuh"
#include "fx64.cuh"

using namespace jfnk;
typedef long double Q;

// r: contributions over 3 h / 16 as elem_vjp3; mag: the sum of the magnitudes of the largest one's terms
static void reference(const double u[8], const double w[8], Q kap, Q r[8], Q& mag) {
    const Q a = 1 / (2 * std::sqrt((Q)3));
    Q m[8];
    for (int c = 0; c < 8; ++c) r[c] = m[c] = 0;
    for (int q = 0; q < 8; ++q) {
        Q N[8], G[8][3], uq = 0, gu[3] = {0, 0, 0}, gw[3] = {0, 0, 0};
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
            uq += N[c] * u[c];
            for (int d = 0; d < 3; ++d) {
                gu[d] += G[c][d] * u[c];
                gw[d] += G[c][d] * w[c];
            }
        }
        const Q k = kap / 8 * 16 / 3;
        for (int c = 0; c < 8; ++c)
            for (int d = 0; d < 3; ++d) {
                const Q f = k * (1 + uq * uq) * gw[d] * G[c][d], s = k * 2 * uq * gu[d] * gw[d] * N[c];
                r[c] += f + s;
                m[c] += std::fabs(f) + std::fabs(s);
            }
    }
    mag = *std::max_element(m, m + 8);
}

static bool fixed(const double u[8], const double w[8], double kap, double scale, double r[8]) {
    fx_t p[8], q[8], ri[8];
    int xu = 0, xw = 0, X = 0;
    for (int c = 0; c < 8; ++c) {
        p[c] = fx_pack(u[c]);
        q[c] = fx_pack(w[c]);
        xu = std::max(xu, fx_exp(p[c]));
        xw = std::max(xw, fx_exp(q[c]));
    }
    if (xu >= kFxMaxExp || !fx_exp_ok(xw) || !fx_scale_ok(kap)) return false;
    fx_vjp3(p, xu, q, xw, kap == 1.0 ? fx_scale(scale) : fx_scale_kappa(fx_scale(scale), kap), ri, X);
    for (int c = 0; c < 8; ++c) r[c] = fx_to_double(ri[c], X);
    return true;
}

static std::mt19937_64 rng(11);
static double uni() { return std::uniform_real_distribution<double>(-1, 1)(rng); }
static double nrm() { return std::normal_distribution<double>()(rng); }

static double corner(int size, int sign, int c, int ex) {
    const double m = size == 0 ? 1 - 0x1p-53 : size == 1 ? 0.5 + 0.5 * std::fabs(uni())
                     : size == 2 ? std::ldexp(1.0, -(int)(rng() % 40)) * 0.999
                     : size == 3 ? 1 - 1e-11 * std::fabs(uni()) : std::fabs(uni());
    return std::ldexp((sign >> c & 1) ? -m : m, ex);
}

int main() {
    int bad = 0, cases = 0;
    const double scale = 3.0 / 16 / 100;
    const int eu[] = {-1000, -400, -299, -120, -40, -8, -2, -1, 0, 1, 2, 9, 30, 53}, ew[] = {-299, -40, -1, 0, 1, 30, 53};
    for (int a : eu)
        for (int b : ew)
            for (int size = 0; size < 25; ++size)
                for (int sign = 0; sign < 256; sign += 1 + (size % 5 != 0) * (int)(rng() % 9)) {
                    const double kap = size % 5 == 4 ? std::exp(60 * uni()) : 1.0;
                    const int sw = size < 5 ? sign : (int)(rng() & 255);
                    double u[8], w[8], r[8];
                    for (int c = 0; c < 8; ++c) {
                        u[c] = corner(size % 5, sign, c, a);
                        w[c] = corner(size / 5, sw, c, b);
                    }
                    w[sign & 7] = std::ldexp(w[sign & 7] < 0 ? -0.75 : 0.75, b);
                    Q q[8], mag, err = 0;
                    reference(u, w, (Q)kap * scale, q, mag);
                    ++cases;
                    if (!fixed(u, w, kap, scale, r)) {
                        printf("refused: %d %d size %d\n", a, b, size), ++bad;
                        continue;
                    }
                    for (int c = 0; c < 8; ++c) err = std::max(err, std::fabs(q[c] - r[c]));
                    if (!(err <= 0x1p-44L * mag)) printf("%d %d size %d sign %d: %Lg of %Lg\n", a, b, size, sign, err, mag), ++bad;
                }
    const double out[] = {INFINITY, -INFINITY, NAN, 0x1p54, -1e300};
    for (double x : out) {
        const double o[8] = {0, 0, 0, x, 0, 0, 0, 0}, in[8] = {1, 0, 1, 1, 1, 1, 1, 1};
        double r[8];
        ++cases;
        if (fixed(o, in, 1.0, scale, r) || fixed(in, o, 1.0, scale, r)) printf("taken: %g\n", x), ++bad;
    }
    const int m = 5;
    for (int kind = 0; kind < 9; ++kind)
        for (int kw = 0; kw < 3; ++kw) {
            Q e64 = 0, efx = 0;
            for (int trial = 0; trial < 20; ++trial) {
                const int n = kind == 0 ? 16 : kind == 1 ? 64 : kind == 2 ? 256 : 128;
                double o[3];
                for (double& x : o) x = 0.5 * (uni() + 1) * (1 - m / (double)n);
                const int N = (m + 1) * (m + 1) * (m + 1);
                std::vector<double> U(N), W(N), A(N, 0), B(N, 0);
                std::vector<Q> R(N, 0);
                auto id = [&](int x, int y, int z) { return (z * (m + 1) + y) * (m + 1) + x; };
                for (int z = 0; z <= m; ++z)
                    for (int y = 0; y <= m; ++y)
                        for (int x = 0; x <= m; ++x) {
                            auto f = [&](double s) { return std::sin(M_PI * s); };
                            const double s = f(o[0] + x / (double)n) * f(o[1] + y / (double)n) * f(o[2] + z / (double)n);
                            const double v[] = {s, s, s, s + 0.1 * nrm(), uni(), 1e-8 * s, 1e3 * s, 1 + 1e-9 * nrm(), 1e-30 * nrm()};
                            U[id(x, y, z)] = v[kind];
                            W[id(x, y, z)] = kw == 0 ? f(o[1] + 2 * x / (double)n) * f(o[0] + y / (double)n) + z / (double)n
                                             : kw == 1 ? nrm() : 1e-20 * uni();
                        }
                for (int z = 0; z < m; ++z)
                    for (int y = 0; y < m; ++y)
                        for (int x = 0; x < m; ++x) {
                            double u[8], w[8], a[8], b[8], dk;
                            Q q[8], mag;
                            for (int c = 0; c < 8; ++c) {
                                u[c] = U[id(x + (c & 1), y + (c >> 1 & 1), z + (c >> 2))];
                                w[c] = W[id(x + (c & 1), y + (c >> 1 & 1), z + (c >> 2))];
                            }
                            const double kap = trial & 1 ? std::exp(0.7 * nrm()) : 1.0;
                            reference(u, w, (Q)kap * scale, q, mag);
                            elem_vjp3<double>(u, w, kap, a, dk);
                            if (!fixed(u, w, kap, scale, b)) printf("refused: field %d\n", kind), ++bad;
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
            if (getenv("FX_PRINT")) printf("field %d %d: %Lg against %Lg\n", kind, kw, std::sqrt(efx), std::sqrt(e64));
            if (!(efx <= 1.5L * 1.5L * e64)) printf("field %d %d: %Lg against %Lg\n", kind, kw, std::sqrt(efx), std::sqrt(e64)), ++bad;
        }
    if (!bad) printf("ok %d\n", cases);
    return bad != 0;
}
