// Host check of the factorised Neo-Hookean element (csrc/fx_beam.cuh) against a
// long double quadrature and the plain FP64 element (csrc/element.cuh); built
// with -fsanitize=signed-integer-overflow.
//   1. ln J and 1 / J over their range: 2^-54 (absolute) and 2^-52 (relative).
//   2. elements stretched, bent, twisted by a large rotation, with displacement
//      noise up to 0.4 h: the error's 2-norm over 3000 elements is at most that
//      of the FP64 element.
//   3. what is left to FP64: J <= 0, non-finite and huge displacements.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <random>

#include "element.cuh"
#include "fx_beam.cuh"

using namespace jfnk;
typedef long double Q;
static std::mt19937_64 rng(5);
static double uni() { return std::uniform_real_distribution<double>(-1, 1)(rng); }

static void reference(const double* u, double inv_h, Q* r) {
    const Q A = 1 / (2 * std::sqrt((Q)3)), ih = inv_h, w = 1 / (8 * ih * ih * ih);
    for (int k = 0; k < 24; ++k) r[k] = 0;
    for (int q = 0; q < 8; ++q) {
        Q g[8][3], F[3][3] = {{1, 0, 0}, {0, 1, 0}, {0, 0, 1}}, C[3][3];
        for (int c = 0; c < 8; ++c) {
            Q l[3], s[3];
            for (int d = 0; d < 3; ++d) {
                const Q p = (q >> d & 1) ? (Q)0.5 + A : (Q)0.5 - A;
                l[d] = (c >> d & 1) ? p : 1 - p;
                s[d] = (c >> d & 1) ? ih : -ih;
            }
            g[c][0] = s[0] * l[1] * l[2];
            g[c][1] = s[1] * l[0] * l[2];
            g[c][2] = s[2] * l[0] * l[1];
            for (int i = 0; i < 3; ++i)
                for (int d = 0; d < 3; ++d) F[i][d] += ((Q)u[3 * c + i] - u[i]) * g[c][d];
        }
        for (int i = 0; i < 3; ++i)
            for (int d = 0; d < 3; ++d) {
                const int a = (i + 1) % 3, b = (i + 2) % 3, e = (d + 1) % 3, f = (d + 2) % 3;
                C[i][d] = F[a][e] * F[b][f] - F[a][f] * F[b][e];
            }
        const Q J = F[0][0] * C[0][0] + F[0][1] * C[0][1] + F[0][2] * C[0][2];
        const Q kc = ((Q)kBeamLambda * std::log(J) - (Q)kBeamMu) / J;
        for (int c = 0; c < 8; ++c)
            for (int i = 0; i < 3; ++i)
                for (int d = 0; d < 3; ++d) r[3 * c + i] += w * ((Q)kBeamMu * F[i][d] + kc * C[i][d]) * g[c][d];
    }
}

int main() {
    int bad = 0;
    for (int i = 0; i < 400000; ++i) {
        const double x = (i & 1) ? 1 + 0.5 * uni() : std::exp(11 * uni());
        fx_t l;
        double rc;
        if (!fx_log_rcp(x, l, rc)) { printf("refused %g\n", x), ++bad; continue; }
        if (!(std::fabs(std::ldexp((Q)l, -57) - std::log((Q)x)) < 0x1p-54L)) printf("ln %.17g\n", x), ++bad;
        if (!(std::fabs((Q)rc * x - 1) < 0x1p-52L)) printf("1/%.17g\n", x), ++bad;
    }
    for (double x : {0.0, -1.0, 1e-9, 1e9, (double)INFINITY, (double)NAN}) {
        fx_t l;
        double rc;
        if (fx_log_rcp(x, l, rc)) printf("taken %g\n", x), ++bad;
    }
    for (int kind = 0; kind < 6; ++kind) {
        Q e64 = 0, efx = 0;
        for (int t = 0; t < 3000; ++t) {
            const double n = kind == 0 ? 1 : kind == 1 ? 4 : 16;
            const double o[3] = {10 * std::fabs(uni()), std::fabs(uni()), std::fabs(uni())}, th = 0.25 * o[0];
            double u[24], a[24], b[24];
            Q q[24];
            for (int c = 0; c < 8; ++c) {
                const double x = o[0] + (c & 1) / n, y = o[1] + ((c >> 1) & 1) / n - 0.5, z = o[2] + (c >> 2) / n - 0.5;
                const bool twist = kind >= 4;
                u[3 * c] = twist ? 0 : 0.02 * x;
                u[3 * c + 1] = twist ? y * std::cos(th) - z * std::sin(th) - y : 0.05 * std::sin(0.3 * x);
                u[3 * c + 2] = twist ? y * std::sin(th) + z * std::cos(th) - z : 0;
                const double noise = kind == 3 ? 0.4 : kind == 4 ? 0.0 : 0.2;
                for (int i = 0; i < 3; ++i) u[3 * c + i] += noise / n * uni();
            }
            reference(u, n, q);
            elem_neohooke<double>(u, n, a);
            const bool ok = fx_neohooke(u, fx_beam(n), b);
            bool fine = true;
            for (int k = 0; k < 24; ++k) fine = fine && std::isfinite((double)q[k]);
            if (ok != fine) printf("kind %d: taken %d, finite %d\n", kind, ok, fine), ++bad;
            if (!ok || !fine) continue;
            for (int k = 0; k < 24; ++k) {
                e64 += (a[k] - q[k]) * (a[k] - q[k]);
                efx += (b[k] - q[k]) * (b[k] - q[k]);
            }
        }
        if (!(efx <= e64)) printf("kind %d: %Lg against %Lg\n", kind, std::sqrt(efx), std::sqrt(e64)), ++bad;
    }
    for (double x : {-3.0, 1e20, (double)INFINITY, (double)NAN}) {
        double u[24] = {0}, r[24];
        u[21] = x;
        if (fx_neohooke(u, fx_beam(1.0), r)) printf("taken with %g\n", x), ++bad;
    }
    if (!bad) printf("ok\n");
    return bad != 0;
}
