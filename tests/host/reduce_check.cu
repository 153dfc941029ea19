// GPU check of the reductions' device functions (csrc/reduce.cuh, stencil.cuh,
// coarse.cuh) and of the batched norms (csrc/batch.cu), which no entry point
// reaches on chosen values:
//   1. warp_sum(double): mixed exponents, cancellation, zeros and subnormals, the
//      ends of its integer path, NaN and infinities in one lane;
//   2. set_eps_slot: the norm, the FD step and its reciprocal as IEEE square
//      root and divisions give them, over the exponent range;
//   3. batched FP32 norms over values whose squares leave FP32's range;
//   4. coarse_rsqrt in FP32: 1 / sqrt of a sum of squared norms, rounded once.
// Prints one line per violation and "ok" at the end.
#include <cmath>
#include <cstdio>
#include <cstring>
#include <random>
#include <vector>

#include "batch.cuh"
#include "coarse.cuh"
#include "reduce.cuh"
#include "stencil.cuh"

using namespace jfnk;

static int bad = 0;
#define CHECK(cond, ...)         \
    do {                         \
        if (!(cond)) {           \
            if (bad++ < 20) {    \
                printf(__VA_ARGS__); \
                printf("\n");    \
            }                    \
        }                        \
    } while (0)

template <typename T>
struct Dev {
    T* p = nullptr;
    size_t n;
    explicit Dev(size_t count) : n(count) {
        cudaMalloc(&p, n * sizeof(T));
        cudaMemset(p, 0, n * sizeof(T));
    }
    explicit Dev(const std::vector<T>& v) : Dev(v.size()) { cudaMemcpy(p, v.data(), n * sizeof(T), cudaMemcpyHostToDevice); }
    ~Dev() { cudaFree(p); }
    std::vector<T> get() const {
        std::vector<T> v(n);
        cudaMemcpy(v.data(), p, n * sizeof(T), cudaMemcpyDeviceToHost);
        return v;
    }
};

// ---- 1 --------------------------------------------------------------------
__global__ void warp_sum_kernel(const double* x, double* out) {
    const double s = warp_sum(x[blockIdx.x * 32 + threadIdx.x]);
    out[blockIdx.x * 32 + threadIdx.x] = s;
}

static void check_warp_sum() {
    std::mt19937_64 rng(1);
    std::uniform_real_distribution<double> u(-1.0, 1.0);
    std::vector<double> x;
    auto warp = [&](auto f) {
        for (int l = 0; l < 32; ++l) x.push_back(f(l));
    };
    for (int r = 0; r < 50; ++r) {
        warp([&](int) { return u(rng); });
        warp([&](int) { return std::ldexp(u(rng), (int)(rng() % 120) - 60); });
        warp([&](int) { return std::fabs(std::ldexp(u(rng), (int)(rng() % 12))); });
        warp([&](int) { return std::ldexp(u(rng), -960 - (int)(rng() % 120)); });   // both sides of the lower end
        warp([&](int) { return std::ldexp(u(rng), 1010 + (int)(rng() % 10)); });    // and of the upper
        double a[16];
        for (double& v : a) v = std::ldexp(u(rng), (int)(rng() % 40));
        warp([&](int l) { return l < 16 ? a[l] : -a[31 - l]; });                    // cancels to zero
        warp([&](int l) { return l == 7 ? u(rng) : 0.0; });
        warp([&](int l) { return l == 3 ? 1.0 : 4.9406564584124654e-324; });
    }
    warp([](int) { return 0.0; });
    warp([](int) { return -0.0; });
    warp([](int) { return 4.9406564584124654e-324; });
    warp([](int) { return 1.7976931348623157e308; });  // overflows
    const size_t finite = x.size() / 32;
    for (double v : {std::nan(""), (double)INFINITY, -(double)INFINITY}) warp([&](int l) { return l == 19 ? v : 1.0; });
    Dev<double> dx(x), dy(x.size());
    warp_sum_kernel<<<(int)(x.size() / 32), 32>>>(dx.p, dy.p);
    const std::vector<double> y = dy.get();
    for (size_t w = 0; w < x.size() / 32; ++w) {
        for (int l = 1; l < 32; ++l) CHECK(memcmp(&y[w * 32], &y[w * 32 + l], 8) == 0, "warp %zu: lanes differ", w);
        const double got = y[w * 32];
        if (w >= finite) {
            const double v = x[w * 32 + 19];
            CHECK(std::isnan(v) ? std::isnan(got) : got == v, "warp %zu: %g instead of %g", w, got, v);
            continue;
        }
        long double s = 0, most = 0;
        for (int l = 0; l < 32; ++l) {
            s += (long double)x[w * 32 + l];
            most = std::fmax(most, std::fabs((long double)x[w * 32 + l]));
        }
        if (std::fabs(s) > 1.7976931348623157e308L) {
            CHECK(std::isinf(got), "warp %zu: %g instead of an overflow", w, got);
            continue;
        }
        // a lane loses less than 2^-5 of the last place of the largest, and the result is rounded
        // once; outside of the integer path five rounded additions of partial sums
        const long double tol = std::fmax(std::ldexp(most * 32, -53) * 5, 4.95e-324L);
        const bool ints = most >= std::ldexp(1.0L, 64 - 1023) && most < std::ldexp(1.0L, 2041 - 1023);
        const long double fine = std::ldexp(most, -52) + std::ldexp(std::fabs(s), -53);
        CHECK(std::fabs(got - s) <= (ints ? fine : tol), "warp %zu: %.17g, off by %Lg", w, got, (long double)got - s);
    }
}

// ---- 2 --------------------------------------------------------------------
__global__ void eps_kernel(const double* tot, const double* k, int n, int unit, EpsSlot* slot, double* nrm) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) set_eps_slot(slot + i, EpsPre{k[i], 1.0 / k[i]}, tot[i], unit != 0, nullptr, nrm + i);
}

static void check_eps_slot() {
    std::mt19937_64 rng(2);
    std::uniform_real_distribution<double> u(1.0, 2.0);
    std::vector<double> tot, k;
    for (int i = 0; i < 400000; ++i) {
        const int wide = i & 1;
        tot.push_back(std::ldexp(u(rng), wide ? (int)(rng() % 2040) - 1020 : (int)(rng() % 60) - 30));
        k.push_back(std::ldexp(u(rng), wide ? (int)(rng() % 60) - 40 : -26));
    }
    for (double t : {1.0, 4.0, 0x1.fffffffffffffp+1, 0x1.0000000000001p+0, 4.9406564584124654e-324}) {
        tot.push_back(t);
        k.push_back(1.4901161193847656e-08);
    }
    const int n = (int)tot.size();
    Dev<double> dt(tot), dk(k), dn(n);
    Dev<EpsSlot> ds(n);
    for (int unit = 0; unit < 2; ++unit) {
        eps_kernel<<<(n + 255) / 256, 256>>>(dt.p, dk.p, n, unit, ds.p, dn.p);
        const std::vector<double> nrm = dn.get();
        const std::vector<EpsSlot> s = ds.get();
        for (int i = 0; i < n; ++i) {
            const double r = std::sqrt(tot[i]), e = k[i] / r, inv = unit ? 1.0 / k[i] : 1.0 / e;
            CHECK(nrm[i] == r, "norm of %a: %a instead of %a", tot[i], nrm[i], r);
            CHECK(s[i].e == e, "step %a / %a: %a instead of %a", k[i], r, s[i].e, e);
            CHECK(s[i].inv == inv, "reciprocal step: %a instead of %a", s[i].inv, inv);
            CHECK(s[i].ef == (float)e && s[i].invf == (float)inv, "FP32 step of %a", e);
        }
    }
}

// ---- 3 --------------------------------------------------------------------
static void check_batched_norms() {
    std::mt19937_64 rng(3);
    std::uniform_real_distribution<double> u(0.5, 1.0);
    const int n = 70, kinds = 5;
    const double scale[kinds] = {1.0, 1e-25, 1e-19, 3e19, 1e37};
    const Grid g = Grid::make(2, n);
    for (int what = 0; what < 2; ++what) {
        std::vector<BVec> d;
        std::vector<BSeg> segs;
        std::vector<std::vector<float>> x(kinds);
        std::vector<Dev<float>*> dx;
        Dev<double> out(kinds);
        Dev<double> partial((size_t)kinds * 2 * kMaxRedBlocks);
        Dev<unsigned int> counter(kinds);
        int blocks = 0;
        for (int q = 0; q < kinds; ++q) {
            for (long long i = 0; i < g.size; ++i) x[q].push_back((float)(scale[q] * u(rng) * (i % 3 == 0 ? -1 : 1)));
            dx.push_back(new Dev<float>(x[q]));
            BVec v;
            memset(&v, 0, sizeof(v));
            v.g = g;
            v.x = dx[q]->p;
            v.what = what;
            v.out = out.p + q;
            v.partials = partial.p + (size_t)q * 2 * kMaxRedBlocks;
            v.counter = counter.p + q;
            d.push_back(v);
            const int nb = 1 + q;
            segs.push_back(BSeg{blocks, nb, 0, 0});
            blocks += nb;
        }
        Dev<BVec> dd(d);
        Dev<BSeg> dsg(segs);
        CHECK(launch_bvec<float>(BOp::STAT, dd.p, dsg.p, kinds, blocks, 0) == JFNK_OK, "launch");
        const std::vector<double> got = out.get();
        for (int q = 0; q < kinds; ++q) {
            long double s = 0;
            for (long long i = 0; i < g.size; ++i)
                if (grid_unknown(g, i)) s += what ? (long double)x[q][i] * x[q][i] : std::fabs((long double)x[q][i]);
            if (what) s = std::sqrt(s);
            // at most 20 entries a thread, 5 + 3 levels, 5 blocks: below 40 roundings
            CHECK(std::fabs(got[q] - s) <= std::ldexp(40 * s, -53), "batched statistic %d at %g: %.17g, off by %Lg of it",
                  what, scale[q], got[q], (got[q] - s) / s);
        }
        for (auto* p : dx) delete p;
    }
}

// ---- 4 --------------------------------------------------------------------
__global__ void rsqrt_kernel(const float* p, int n, int count, float* out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < count) out[i] = coarse_rsqrt(p + (size_t)i * n, n);
}

static void check_coarse_rsqrt() {
    std::mt19937_64 rng(4);
    std::uniform_real_distribution<double> u(0.0, 1.0);
    const int count = 100000;
    for (int n : {1, 2, 7, 15}) {
        std::vector<float> p;
        for (int i = 0; i < count; ++i) {
            const int e = (int)(rng() % 240) - 130;
            for (int w = 0; w < n; ++w) p.push_back((float)std::ldexp(u(rng), e - (int)(rng() % 8)));
            p.back() = std::fmax(p.back(), 0x1p-126f);
        }
        Dev<float> dp(p), dy(count);
        rsqrt_kernel<<<(count + 255) / 256, 256>>>(dp.p, n, count, dy.p);
        const std::vector<float> y = dy.get();
        for (int i = 0; i < count; ++i) {
            long double s = 0;
            for (int w = 0; w < n; ++w) s += (long double)p[(size_t)i * n + w];
            const long double want = 1 / std::sqrt(s);
            int e;
            std::frexp((double)want, &e);
            // the start is within 2 ulp (e below 2^-21): the step leaves 3/8 e^2 and three
            // roundings of e, together below 2^-43 of the result
            const long double ulp = std::ldexp(1.0L, e - 24);
            CHECK(std::fabs(y[i] - want) <= (0.5L + 0x1p-18L) * ulp, "1/sqrt of %Lg: off by %Lg ulp", s, (y[i] - want) / ulp);
        }
    }
}

int main() {
    check_coarse_rsqrt();
    check_warp_sum();
    check_eps_slot();
    check_batched_norms();
    const cudaError_t e = cudaDeviceSynchronize();
    CHECK(e == cudaSuccess, "%s", cudaGetErrorString(e));
    if (bad == 0) printf("ok\n");
    return bad == 0 ? 0 : 1;
}
